// Tensor-core products of the correction network's training step: the hidden layers' forward
// products, the deltas back through W2 and W3, and the weight gradients of W1, W2 and W3.
//
// Precision: every FP32 operand is split into three BF16 parts, x = hi + mid + lo (exact: each
// part takes the next 8 bits of the significand, and BF16 has the FP32 exponent range), and a
// product takes the six part pairs down to 2^-16 (hi hi, hi mid, mid hi, hi lo, lo hi, mid mid):
// what is dropped is below 2^-24 of the product, so the result has FP32 accuracy with the FP32
// accumulation of tcgen05.mma kind::f16 (BF16 operands).  That accumulation truncates, once for every
// product added to a sum.  The weight gradients, whose sums run over the batch, therefore have the hi hi
// products in one accumulator and the others, 2^-8 and less of them, in a second: one truncation of the
// sum's size per chunk instead of six.  Error of dW2 against FP64 at 8192 rows, 35 chunks a sum: 5.3e-6 with
// one accumulator, 2.8e-6 with two (and 3.6e-6 with one and 14 chunks a sum, at 158 us a step instead of
// 143); 2.4e-6 of it is there at 256 rows.
//
// Operand layout in global memory ("blocks"): an operand with R rows and K columns is cut into
// blocks of 128 rows x 16 k, block (kc, rb) at ((kc * nRB + rb) * 12 KB), each the three parts
// (4 KB each) in the K-major canonical layout of 8-row x 16-byte core matrices (128 bytes apart
// along K, 256 along the rows).  Rows beyond R and k beyond K are zero.  Every activation and delta
// is written in this layout both ways by the kernel that makes it: rows = its rows (the operand of a
// layer's product) and rows = its columns (the operand of a weight gradient, K = the batch).
//
// A step is nine launches: pack_x (the batch's inputs), three forward products, out_train (output layer,
// loss, deltas of layer 3), two products back, the three weight gradients in one launch, and step_finish
// (sums of the gradient's partial products, Adam, the next step's weight operands).  In seventeen launches, with FP32 deltas
// packed in passes of their own and each gradient summed by a launch, a step of 8192 rows took 200 us and one of
// 1024 rows 173; now 144 and 88 (hidden 256, back to back).  What bounds it: the launches' latencies in
// line, about 8 us each, and at 8192 rows the epilogues.
//
// mlp_gemm3_kernel: C(m, n) = sum_k A(m, k) B(n, k) over one slice of K, one 128 x TN tile per
// CTA; warp 0 streams the blocks with 1-D bulk copies into six stages, warp 1 issues the six
// MMAs per 16-k chunk into TMEM, warps 2..9 read the tile and apply the epilogue: store a partial
// product (weight gradients, summed over slices afterwards), bias + tanh (forward) or times
// 1 - H^2 (back through tanh), and write the result also as the next products' operands (row and
// transposed, staged in the idle pipeline buffers) and its column sums.  Every wait is bounded.
// What bounds a layer's product is the epilogue (tanh and the three-part split of each value, twice).  TN = 32
// spreads it over four times the CTAs as long as these are at most two per SM: 4096 rows, 107 us a step against
// 125 with TN = 128 (64: 114), 1024 rows 88 / 113 (99); at 8192 rows the operands read four times as often cost
// more, 172 / 144 (147).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "gw_internal.cuh"
#include "ptx.cuh"

namespace gw {

namespace {

constexpr int TR = 128;                    // rows of a block, and each side of a tile
constexpr int NPL = 3;                     // BF16 parts: hi, mid, lo
constexpr uint32_t PLB = TR * 16 * 2;      // 4 KB: one part of one block
constexpr uint32_t BLK = NPL * PLB;        // 12 KB: one block
constexpr int STAGES = 6;
// a stage: a block of A and TN rows of one of B
constexpr uint32_t stage_bytes(int tn) { return BLK + NPL * tn * 32; }
constexpr size_t smem_bytes(int tn) { return STAGES * stage_bytes(tn) + 256; }
constexpr int NEPI = 8;                    // epilogue warps: two per TMEM lane quarter
constexpr int NTHREADS = (2 + NEPI) * 32;  // warp 0 copies, warp 1 MMAs, warps 2..9 epilogue
constexpr uint64_t DRAIN_NS = 2000000000ull;
constexpr int X_ROWS = 32, X_MAX_IN = 64;  // rows of a pack_x CTA; the most inputs a network has
constexpr int OUT_ROWS = 16;               // rows of an out_train CTA: one k chunk of the transposed deltas

__host__ __device__ constexpr uint32_t blk_off(int r, int k)  // r < 128, k < 16
{
    return (r >> 3) * 256 + ((k >> 3) & 1) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ void named_bar_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

__device__ __forceinline__ void split3(float x, uint16_t &h, uint16_t &m, uint16_t &l)
{
    const __nv_bfloat16 bh = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(bh);
    const __nv_bfloat16 bm = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(bm);
    h = __bfloat16_as_ushort(bh);
    m = __bfloat16_as_ushort(bm);
    l = __bfloat16_as_ushort(__float2bfloat16_rn(r2));
}

// 16 values of one row into the three parts of a block (k 0..15 of row r)
__device__ __forceinline__ void store_row16(uint8_t *blk, int r, const float *v)
{
    uint32_t w[NPL][8];
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        uint16_t h0, m0, l0, h1, m1, l1;
        split3(v[e], h0, m0, l0);
        split3(v[e + 1], h1, m1, l1);
        w[0][e >> 1] = h0 | ((uint32_t)h1 << 16);
        w[1][e >> 1] = m0 | ((uint32_t)m1 << 16);
        w[2][e >> 1] = l0 | ((uint32_t)l1 << 16);
    }
#pragma unroll
    for (int p = 0; p < NPL; ++p) {
        *reinterpret_cast<uint4 *>(blk + p * PLB + blk_off(r, 0)) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
        *reinterpret_cast<uint4 *>(blk + p * PLB + blk_off(r, 8)) = make_uint4(w[p][4], w[p][5], w[p][6], w[p][7]);
    }
}

// Eight values of one row (k 8 h .. 8 h + 7 of a chunk) into the three parts of a block.
__device__ __forceinline__ void store_row8(uint8_t *blk, int r, int h, const float *v)
{
    uint32_t w[NPL][4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
        uint16_t h0, m0, l0, h1, m1, l1;
        split3(v[e], h0, m0, l0);
        split3(v[e + 1], h1, m1, l1);
        w[0][e >> 1] = h0 | ((uint32_t)h1 << 16);
        w[1][e >> 1] = m0 | ((uint32_t)m1 << 16);
        w[2][e >> 1] = l0 | ((uint32_t)l1 << 16);
    }
#pragma unroll
    for (int p = 0; p < NPL; ++p)
        *reinterpret_cast<uint4 *>(blk + p * PLB + blk_off(r, 8 * h)) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
}

// The inputs of a batch, rows X[rows ? rows[r] : r], as the row operand (R x C) and, if colop is given, as the
// transposed one (rows c, k = r), whose rows beyond C are never written: the buffer is cleared once.
__global__ void __launch_bounds__(128) pack_x_kernel(const float *__restrict__ X, const int *__restrict__ rows, int R,
                                                     int C, uint8_t *__restrict__ rowop, uint8_t *__restrict__ colop)
{
    __shared__ float tile[X_ROWS][X_MAX_IN + 1];
    const int r0 = blockIdx.x * X_ROWS, t = threadIdx.x, nrb = (R + TR - 1) / TR, nkc = (C + 15) / 16;
    for (int e = t; e < X_ROWS * 16 * nkc; e += 128) {
        const int i = e / (16 * nkc), c = e - i * 16 * nkc, r = r0 + i;
        tile[i][c] = r < R && c < C ? X[(long)(rows ? rows[r] : r) * C + c] : 0.f;
    }
    __syncthreads();
    for (int e = t; e < X_ROWS * nkc * 2; e += 128) {
        const int i = e % X_ROWS, u = e / X_ROWS, r = r0 + i;  // u: eight columns
        store_row8(rowop + ((size_t)(u >> 1) * nrb + (r >> 7)) * BLK, r & 127, u & 1, &tile[i][8 * u]);
    }
    if (colop)
        for (int e = t; e < C * (X_ROWS / 16); e += 128) {
            const int c = e % C, j = e / C;
            if (r0 + 16 * j >= R)
                continue;
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] = tile[16 * j + i][c];
            store_row16(colop + (size_t)((r0 >> 4) + j) * BLK, c, v);
        }
}

// The 2-wide output layer of a training step over OUT_ROWS rows: y = W4 h + b4 (h = H2[b]), d4 = (y - t) / B, the deltas of layer 3, D[b][n] = (d4 W4)[n] (1 - h[n]^2), as row and
// transposed operand, their column sums (csum[block][n]) and the block's share of the output layer's gradient and of
// the loss, part[block] = [sum_b d4 h^T (2 x Hd) | sum_b d4 | sum_b |y - t|^2] (2 Hd + 3 values).
__global__ void __launch_bounds__(256) out_train_kernel(const float *__restrict__ H2, int Hd,
                                                        const __half *__restrict__ W4, const float *__restrict__ b4,
                                                        int batch, const float *__restrict__ T,
                                                        const int *__restrict__ trow, float invB,
                                                        uint8_t *__restrict__ rowop, uint8_t *__restrict__ colop,
                                                        float *__restrict__ csum, float *__restrict__ part)
{
    extern __shared__ float hs[];  // [OUT_ROWS][pitch]
    __shared__ float d4[OUT_ROWS][2], l2[OUT_ROWS];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, b0 = blockIdx.x * OUT_ROWS;
    const int nkc = (Hd + 15) / 16, pitch = 16 * nkc + 1, nrb = (batch + TR - 1) / TR;
    const float c0 = b4[0], c1 = b4[1];
#pragma unroll
    for (int r = warp; r < OUT_ROWS; r += 8) {
        const int b = b0 + r;
        float y0 = 0.f, y1 = 0.f, t0 = 0.f, t1 = 0.f;
        if (b < batch) {  // before the products: two dependent loads
            const long q = trow ? trow[b] : b;
            t0 = T[2 * q];
            t1 = T[2 * q + 1];
        }
        for (int n = lane; n < 16 * nkc; n += 32) {
            const float hv = b < batch && n < Hd ? H2[(long)b * Hd + n] : 0.f;
            hs[r * pitch + n] = hv;
            if (n < Hd) {
                y0 = fmaf(__half2float(W4[n]), hv, y0);
                y1 = fmaf(__half2float(W4[Hd + n]), hv, y1);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            y0 += __shfl_xor_sync(0xffffffffu, y0, o);
            y1 += __shfl_xor_sync(0xffffffffu, y1, o);
        }
        if (lane == 0) {
            float e0 = 0.f, e1 = 0.f;
            if (b < batch) {
                e0 = y0 + c0 - t0;
                e1 = y1 + c1 - t1;
            }
            d4[r][0] = e0 * invB;
            d4[r][1] = e1 * invB;
            l2[r] = e0 * e0 + e1 * e1;
        }
    }
    __syncthreads();
    auto delta = [&](int r, int n, float w0, float w1) {
        const float h = hs[r * pitch + n];
        return (d4[r][0] * w0 + d4[r][1] * w1) * (1.f - h * h);
    };
    for (int e = t; e < OUT_ROWS * nkc * 2; e += 256) {  // row operand: eight columns n of one row
        const int r = e % OUT_ROWS, u = e / OUT_ROWS, b = b0 + r;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int n = 8 * u + i;
            v[i] = n < Hd ? delta(r, n, __half2float(W4[n]), __half2float(W4[Hd + n])) : 0.f;
        }
        store_row8(rowop + ((size_t)(u >> 1) * nrb + (b >> 7)) * BLK, b & 127, u & 1, v);
    }
    if (b0 >= batch)  // rows that only pad the last 128-row block
        return;
    const int G = 2 * Hd + 3, nnb = (Hd + TR - 1) / TR;
    for (int n = t; n < nnb * TR; n += 256) {
        float v[16], cs = 0.f, g0 = 0.f, g1 = 0.f;
        const float w0 = n < Hd ? __half2float(W4[n]) : 0.f, w1 = n < Hd ? __half2float(W4[Hd + n]) : 0.f;
#pragma unroll
        for (int r = 0; r < OUT_ROWS; ++r) {
            v[r] = n < Hd ? delta(r, n, w0, w1) : 0.f;
            cs += v[r];
            if (n < Hd) {
                const float h = hs[r * pitch + n];
                g0 = fmaf(d4[r][0], h, g0);
                g1 = fmaf(d4[r][1], h, g1);
            }
        }
        store_row16(colop + ((size_t)blockIdx.x * nnb + (n >> 7)) * BLK, n & 127, v);
        if (n < Hd) {
            csum[(long)blockIdx.x * Hd + n] = cs;
            part[(long)blockIdx.x * G + n] = g0;
            part[(long)blockIdx.x * G + Hd + n] = g1;
        }
    }
    if (t == 0) {
        float s0 = 0.f, s1 = 0.f, l = 0.f;
        for (int r = 0; r < OUT_ROWS; ++r) {
            s0 += d4[r][0];
            s1 += d4[r][1];
            l += l2[r];
        }
        part[(long)blockIdx.x * G + 2 * Hd] = s0;
        part[(long)blockIdx.x * G + 2 * Hd + 1] = s1;
        part[(long)blockIdx.x * G + 2 * Hd + 2] = l;
    }
}

// Element e of weight matrix l (0..2: out x in, row-major) into its row operand (rows = outputs, k = inputs)
// and, for l = 1, 2, its transpose (rows = inputs).  Padding (k beyond in, rows beyond out) is never written:
// the buffers are cleared once.
__device__ __forceinline__ void pack_weight(const MlpWeightPack &p, int l, long e, float x)
{
    const int in = l == 0 ? p.n_in : p.hidden, nrb = (p.hidden + TR - 1) / TR;
    const int o = (int)(e / in), c = (int)(e - (long)o * in);
    uint16_t h, m, lo;
    split3(x, h, m, lo);
    uint8_t *b = p.row[l] + ((size_t)(c >> 4) * nrb + (o >> 7)) * BLK + blk_off(o & 127, c & 15);
    *reinterpret_cast<uint16_t *>(b) = h;
    *reinterpret_cast<uint16_t *>(b + PLB) = m;
    *reinterpret_cast<uint16_t *>(b + 2 * PLB) = lo;
    if (l > 0) {
        uint8_t *bt = p.col[l - 1] + ((size_t)(o >> 4) * nrb + (c >> 7)) * BLK + blk_off(c & 127, o & 15);
        *reinterpret_cast<uint16_t *>(bt) = h;
        *reinterpret_cast<uint16_t *>(bt + PLB) = m;
        *reinterpret_cast<uint16_t *>(bt + 2 * PLB) = lo;
    }
}

// The three weight matrices (flat at w + off[l]) into their operands.
__global__ void pack_weights_kernel(const float *__restrict__ w, MlpWeightPack p)
{
    const long n0 = (long)p.hidden * p.n_in, n1 = (long)p.hidden * p.hidden, total = n0 + 2 * n1;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int l = i < n0 ? 0 : (i < n0 + n1 ? 1 : 2);
        const long e = l == 0 ? i : i - n0 - (l - 1) * n1;
        pack_weight(p, l, e, w[p.off[l] + e]);
    }
}

// The gradient of every parameter from its partial sums, in a fixed order, then (ADAM) the parameter's Adam step, its
// FP16 rounding and the operands of the rounded weights, else the gradient itself.  Blocks below f.nb_w take the weights of
// the hidden layers, a parameter per thread (n_part slices each); the others 32 columns of a bias or of the output layer
// (W4 and b4 are adjacent, the loss follows), eight threads per column with an eighth of the partial rows each.
template <bool ADAM>
__global__ void __launch_bounds__(256) step_finish_kernel(MlpFinish f, MlpWeightPack p)
{
    __shared__ float red[8][33];
    auto apply = [&](long i, float gi, int l, long e) {
        if (!ADAM) {
            f.grad[i] = gi;
            return;
        }
        const float mi = f.b1 * f.m[i] + (1.f - f.b1) * gi;
        const float vi = f.b2 * f.v[i] + (1.f - f.b2) * gi * gi;
        f.m[i] = mi;
        f.v[i] = vi;
        const float t = f.theta[i] - f.lr * (mi * f.c1) / (sqrtf(vi * f.c2) + f.eps);
        f.theta[i] = t;
        const __half t16 = __float2half_rn(t);
        f.theta16[i] = t16;
        const float t32 = __half2float(t16);
        f.w32[i] = t32;
        if (l < 3)
            pack_weight(p, l, e, t32);
    };
    const long n0 = (long)p.hidden * p.n_in, n1 = (long)p.hidden * p.hidden;
    if ((int)blockIdx.x < f.nb_w) {
        for (long i = blockIdx.x * 256L + threadIdx.x; i < n0 + 2 * n1; i += (long)f.nb_w * 256) {
            const int l = i < n0 ? 0 : (i < n0 + n1 ? 1 : 2);
            const long e = l == 0 ? i : i - n0 - (l - 1) * n1, nw = l == 0 ? n0 : n1;
            const float *q = f.part[l] + e;
            float acc = 0.f;
#pragma unroll 8
            for (int z = 0; z < f.n_part[l]; ++z)
                acc += q[z * nw];
            apply(p.off[l] + e, acc, l, e);
        }
        return;
    }
    // columns: biases of the hidden layers, then the output layer
    int b = (int)blockIdx.x - f.nb_w, l = 0;
    const int per = (p.hidden + 31) / 32;
    while (l < 3 && b >= per) {
        b -= per;
        ++l;
    }
    const int width = l < 3 ? p.hidden : 2 * p.hidden + 3, c = threadIdx.x & 31, r0 = threadIdx.x >> 5, col = b * 32 + c;
    const float *q = l < 3 ? f.csum[l] : f.out_part;
    const int rows = l < 3 ? f.n_csum[l] : f.n_out;
    float acc = 0.f;
    if (col < width) {
#pragma unroll 8
        for (int r = r0; r < rows; r += 8)
            acc += q[(long)r * width + col];
    }
    red[r0][c] = acc;
    __syncthreads();
    if (r0 == 0 && col < width) {
        for (int r = 1; r < 8; ++r)
            acc += red[r][c];
        if (l == 3 && col == width - 1) {  // the loss, sum |y - t|^2 / (2B)
            if (f.loss)  // the caller's, and it may collect the steps of several networks and streams
                atomicAdd(f.loss, f.loss_scale * acc);
            return;
        }
        apply((l < 3 ? f.off_b[l] : f.off_out) + col, acc, 3, 0);
    }
}

// Up to three products in one launch; CTA b takes (job, column block, row block, slice of K) in that nesting.
template <int EPI, int TN>
__global__ void __launch_bounds__(NTHREADS, TN < TR ? 2 : 1) mlp_gemm3_kernel(MlpGemmJobs jobs, uint32_t *err, uint64_t wait_ns)
{
    constexpr uint32_t STAGE = stage_bytes(TN), PIPE = STAGES * STAGE, BPL = TN * 32;  // BPL: one part of B's rows
    constexpr int ACC = EPI == 0 ? 2 : 1;  // accumulators: a sum over a batch is a long one (file comment)
    constexpr int PITCH = TN + 1;
    static_assert(TR * PITCH * 4 <= PIPE, "the epilogue stages a tile in the pipeline buffers");
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + PIPE);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(accf + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    volatile int *n_issued = abort_flag + 1;
    volatile int *n_consumed = abort_flag + 2;
    volatile int *epi_ok = abort_flag + 3;  // [NEPI] each epilogue warp's wait result

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int id = blockIdx.x, ji = 0;
    while (ji + 1 < jobs.n && id >= jobs.job[ji].ctas) {
        id -= jobs.job[ji].ctas;
        ++ji;
    }
    const MlpGemmJob &jb = jobs.job[ji];
    const uint8_t *const A = jb.A, *const B = jb.B;
    const int M = jb.M, N = jb.N, nmb = (M + TR - 1) / TR, nnb = (N + TN - 1) / TN, nbb = (N + TR - 1) / TR;
    const int nkc = (jb.K + 15) / 16, nb = id % nnb, mb = id / nnb % nmb, z = id / (nnb * nmb);
    const int k0 = z * jb.kcs, nch = max(0, min(nkc, k0 + jb.kcs) - k0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(accf, 1);
        *abort_flag = 0;
        *n_issued = 0;
        *n_consumed = 0;
        fence_barrier_init();
    }
    if (warp == 1)
        tmem_alloc(tslot, ACC * TN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp == 0) {
        if (lane == 0) {
            for (int i = 0; i < nch; ++i) {
                const int s = i % STAGES;
                if (i >= STAGES && !mbar_wait(&empty[s], ((i / STAGES) - 1) & 1, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_HERK_PRODUCER, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                if (*abort_flag)
                    break;
                uint8_t *st = smem + s * STAGE;
                mbar_arrive_expect_tx(&full[s], STAGE);
                bulk_g2s(st, A + ((size_t)(k0 + i) * nmb + mb) * BLK, BLK, &full[s]);
                const uint8_t *b = B + ((size_t)(k0 + i) * nbb + nb * TN / TR) * BLK + (nb * TN % TR) * 32;
                if (TN == TR) {
                    bulk_g2s(st + BLK, b, BLK, &full[s]);
                } else {
#pragma unroll
                    for (int p = 0; p < NPL; ++p)
                        bulk_g2s(st + BLK + p * BPL, b + p * PLB, BPL, &full[s]);
                }
                *n_issued = i + 1;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t ID = mma_idesc(1, TR, TN, false);  // BF16 x BF16, M 128, N TN
            constexpr uint64_t DP = PLB >> 4, DQ = BPL >> 4, DB = BLK >> 4, DS = STAGE >> 4;
            const uint64_t d0 = smem_desc(smem_u32(smem), 128, 256);
            for (int i = 0; i < nch; ++i) {
                const int s = i % STAGES;
                if (!mbar_wait(&full[s], (i / STAGES) & 1, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_HERK_MMA, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint64_t a = d0 + (uint64_t)s * DS, b = a + DB;
                const uint32_t tx = tmem + (ACC - 1) * TN;
                mma_f16(tmem, a, b, ID, i > 0 ? 1u : 0u);             // hi hi
                mma_f16(tx, a, b + DQ, ID, ACC == 1 || i > 0 ? 1u : 0u);  // hi mid
                mma_f16(tx, a + DP, b, ID, 1);                        // mid hi
                mma_f16(tx, a, b + 2 * DQ, ID, 1);                    // hi lo
                mma_f16(tx, a + 2 * DP, b, ID, 1);                    // lo hi
                mma_f16(tx, a + DP, b + DQ, ID, 1);                   // mid mid
                mma_commit(&empty[s]);
                *n_consumed = i + 1;
            }
            mma_commit(accf);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    } else {
        // epilogue warps 2..9: TMEM lane quarter warp & 3 (one tile row per lane), column half hf
        const int ew = warp - 2, q = warp & 3, hf = ew >> 2, rl = q * 32 + lane, m = mb * TR + rl;
        const int et = ew * 32 + lane;  // 0 .. 255
        const bool wok = __all_sync(0xffffffffu, mbar_wait(accf, 0, wait_ns));
        if (lane == 0) {
            epi_ok[ew] = (wok && *abort_flag == 0) ? 1 : 0;
            if (!wok)
                record_error(err, GW_E_TIMEOUT, SITE_HERK_EPILOGUE, blockIdx.x);
        }
        // every epilogue warp's wait has ended (each is bounded): one decision, from the same votes,
        // for all eight warps, so that all or none of them reach the staging barrier below
        named_bar_sync(1, NEPI * 32);
        bool ok = true;
#pragma unroll
        for (int w = 0; w < NEPI; ++w)
            ok = ok && epi_ok[w] != 0;
        if (!ok) {
            if (lane == 0)
                *abort_flag = 1;
        } else {
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
            // C is null where only the operands are wanted (the deltas)
            float *const C = jb.C;
            const float *const bias = jb.bias, *const H = jb.H;
            uint8_t *const rowop = jb.rowop, *const colop = jb.colop;
            float *const colsum = jb.colsum;
            const long ldc = N, ldh = N;
            float *crow = C + (EPI == 0 ? (long)z * M * N : 0) + (long)m * ldc;
            // 16-byte alignment of every row start of C and H, and of bias
            const bool vec = N % 4 == 0 && ((reinterpret_cast<uintptr_t>(C) | reinterpret_cast<uintptr_t>(bias) |
                                             reinterpret_cast<uintptr_t>(H)) &
                                            15) == 0;
            // the pipeline is idle (every MMA has completed): it stages the tile for colop / colsum
            float *stile = reinterpret_cast<float *>(smem);
            const bool stage = colop || colsum;
            const int nrb_m = (M + TR - 1) / TR, nrb_n = (N + TR - 1) / TR;
            const int nkc_n = (N + 15) / 16, nkc_m = (M + 15) / 16;
            for (int c0 = hf * (TN / 2); c0 < (hf + 1) * (TN / 2); c0 += 16) {
                float v[16];
                if (nch > 0) {
                    tmem_ld16(taddr + c0, v);
                    if (ACC == 2) {
                        float u[16];
                        tmem_ld16(taddr + TN + c0, u);
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            v[e] += u[e];
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        v[e] = 0.f;
                }
                const int n0 = nb * TN + c0;
                if (m < M && vec && n0 + 16 <= N) {
                    // whole 16-column group in range, rows 16-byte aligned: vector loads / stores
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        float4 x = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                        if (EPI == 1) {
                            const float4 b = *reinterpret_cast<const float4 *>(bias + n0 + e);
                            x = make_float4(tanhf(x.x + b.x), tanhf(x.y + b.y), tanhf(x.z + b.z), tanhf(x.w + b.w));
                        } else if (EPI == 2) {
                            const float4 h = *reinterpret_cast<const float4 *>(H + (long)m * ldh + n0 + e);
                            x = make_float4(x.x * (1.f - h.x * h.x), x.y * (1.f - h.y * h.y),
                                            x.z * (1.f - h.z * h.z), x.w * (1.f - h.w * h.w));
                        }
                        if (C)
                            *reinterpret_cast<float4 *>(crow + n0 + e) = x;
                        v[e] = x.x;
                        v[e + 1] = x.y;
                        v[e + 2] = x.z;
                        v[e + 3] = x.w;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int n = n0 + e;
                        float x = 0.f;  // rows and columns out of range stay zero in the packs
                        if (m < M && n < N) {
                            x = v[e];
                            if (EPI == 1)
                                x = tanhf(x + bias[n]);
                            else if (EPI == 2) {
                                const float h = H[(long)m * ldh + n];
                                x *= 1.f - h * h;
                            }
                            if (C)
                                crow[n] = x;
                        }
                        v[e] = x;
                    }
                }
                // this row's 16 values as k chunk n0 / 16 of the row operand (rows m, k = n)
                if (rowop && (n0 >> 4) < nkc_n)
                    store_row16(rowop + ((size_t)(n0 >> 4) * nrb_m + mb) * BLK, rl, v);
                if (stage) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        stile[rl * PITCH + c0 + e] = v[e];
                }
            }
            if (stage) {
                named_bar_sync(1, NEPI * 32);
                // thread et now takes column cl of the tile, chunks JT jh .. JT (jh + 1) - 1 of the transpose
                constexpr int JT = TN * 8 / (NEPI * 32);
                const int cl = et % TN, jh = et / TN, n = nb * TN + cl;
                if (colop)
                    for (int j = JT * jh; j < JT * (jh + 1) && mb * 8 + j < nkc_m; ++j) {
                        float v[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            v[e] = stile[(j * 16 + e) * PITCH + cl];
                        store_row16(colop + ((size_t)(mb * 8 + j) * nrb_n + (n >> 7)) * BLK, n & 127, v);
                    }
                if (colsum && jh == 0 && n < N) {
                    float acc = 0.f;
#pragma unroll 8
                    for (int i = 0; i < TR; ++i)
                        acc += stile[i * PITCH + cl];
                    colsum[(long)mb * N + n] = acc;
                }
            }
        }
    }

    // ---------------- drain: every MMA done, every issued copy landed, then release TMEM
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_wait(accf, 0, DRAIN_NS))
            record_error(err, GW_E_TIMEOUT, SITE_HERK_DRAIN, blockIdx.x);
        const int issued = *n_issued, consumed = *n_consumed;
        for (int i = consumed; i < issued; ++i)
            if (!mbar_wait(&full[i % STAGES], (i / STAGES) & 1, DRAIN_NS)) {
                record_error(err, GW_E_TIMEOUT, SITE_HERK_DRAIN, blockIdx.x);
                break;
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ACC * TN);
    }
}

}  // namespace

size_t mlp_pack3_bytes(int rows, int k)
{
    return (size_t)((rows + TR - 1) / TR) * ((k + 15) / 16) * BLK;
}

cudaError_t launch_mlp_pack_x(const float *X, const int *rows, int R, int C, uint8_t *rowop, uint8_t *colop,
                              cudaStream_t s)
{
    if (R <= 0 || C <= 0 || C > X_MAX_IN)
        return cudaErrorInvalidValue;
    pack_x_kernel<<<(R + TR - 1) / TR * (TR / X_ROWS), 128, 0, s>>>(X, rows, R, C, rowop, colop);
    count_launches(1);
    return cudaGetLastError();
}

int mlp_out_parts(int batch) { return (batch + OUT_ROWS - 1) / OUT_ROWS; }

cudaError_t launch_mlp_out_train(const float *H2, int Hd, const __half *W4, const float *b4, int batch, const float *T,
                                 const int *trow, uint8_t *rowop, uint8_t *colop, float *csum, float *part, cudaStream_t s)
{
    const size_t smem = (size_t)OUT_ROWS * ((Hd + 15) / 16 * 16 + 1) * sizeof(float);
    const cudaError_t e =
        cudaFuncSetAttribute(out_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    out_train_kernel<<<(batch + TR - 1) / TR * (TR / OUT_ROWS), 256, smem, s>>>(H2, Hd, W4, b4, batch, T, trow,
                                                                              1.f / batch, rowop, colop, csum, part);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mlp_pack_weights(const float *w, const MlpWeightPack &p, int num_sms, cudaStream_t s)
{
    const long total = (long)p.hidden * p.n_in + 2L * p.hidden * p.hidden;
    const int blocks = (int)std::max(1L, std::min((total + 255) / 256, 4L * num_sms));
    pack_weights_kernel<<<blocks, 256, 0, s>>>(w, p);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mlp_finish(MlpFinish f, const MlpWeightPack &p, bool adam, int num_sms, cudaStream_t s)
{
    const long total = (long)p.hidden * p.n_in + 2L * p.hidden * p.hidden;
    f.nb_w = (int)std::max(1L, std::min((total + 255) / 256, 8L * num_sms));
    const int grid = f.nb_w + 3 * ((p.hidden + 31) / 32) + (2 * p.hidden + 3 + 31) / 32;
    if (adam)
        step_finish_kernel<true><<<grid, 256, 0, s>>>(f, p);
    else
        step_finish_kernel<false><<<grid, 256, 0, s>>>(f, p);
    count_launches(1);
    return cudaGetLastError();
}

int mlp_gemm3_slices(int K, int splits, int *kcs)
{
    const int nkc = (K + 15) / 16, S0 = std::max(1, std::min(splits, nkc));
    *kcs = (nkc + S0 - 1) / S0;
    return (nkc + *kcs - 1) / *kcs;
}

template <int EPI, int TN>
static cudaError_t launch_gemm3_t(MlpGemmJobs &jobs, uint32_t *err, uint64_t wait_ns, cudaStream_t s)
{
    int ctas = 0;
    for (int i = 0; i < jobs.n; ++i) {
        MlpGemmJob &j = jobs.job[i];
        j.ctas = (j.N + TN - 1) / TN * ((j.M + TR - 1) / TR) * j.slices;
        ctas += j.ctas;
    }
    const cudaError_t e = cudaFuncSetAttribute(mlp_gemm3_kernel<EPI, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem_bytes(TN));
    if (e != cudaSuccess)
        return e;
    mlp_gemm3_kernel<EPI, TN><<<ctas, NTHREADS, smem_bytes(TN), s>>>(jobs, err, wait_ns);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mlp_gemm3(int epi, MlpGemmJobs jobs, int num_sms, uint32_t *err, uint64_t wait_ns, cudaStream_t s)
{
    if (jobs.n < 1 || jobs.n > 3 || epi < 0 || epi > 2)
        return cudaErrorInvalidValue;
    long narrow = 0;  // tiles of 128 x 32
    for (int i = 0; i < jobs.n; ++i) {
        MlpGemmJob &j = jobs.job[i];
        if (j.M <= 0 || j.N <= 0 || j.K <= 0 || (epi == 0 && (j.rowop || j.colop || j.colsum)))
            return cudaErrorInvalidValue;  // partial products are not packed
        if (epi != 0)
            j.slices = mlp_gemm3_slices(j.K, 1, &j.kcs);
        narrow += (long)((j.N + 31) / 32) * ((j.M + TR - 1) / TR);
    }
    if (epi == 0)
        return launch_gemm3_t<0, TR>(jobs, err, wait_ns, s);
    if (narrow <= 2L * num_sms)
        return epi == 1 ? launch_gemm3_t<1, 32>(jobs, err, wait_ns, s) : launch_gemm3_t<2, 32>(jobs, err, wait_ns, s);
    return epi == 1 ? launch_gemm3_t<1, TR>(jobs, err, wait_ns, s) : launch_gemm3_t<2, TR>(jobs, err, wait_ns, s);
}

}  // namespace gw
