// States given as plane-wave coefficients (the DFT input of Sec. 4.1): the transform of each
// periodic part to the real-space grid,
//     u_n(r_j) = N_r^(-1/2) sum_g c_n(g) exp(+2 pi i (m1 j1/n1 + m2 j2/n2 + m3 j3/n3)),
// the discrete form of the paper's u(x) = sum_g u~(g) e^{i g.x} / sqrt(Omega) (unit-norm
// coefficient vectors give unit-norm states on the grid).  The coefficients are scattered into
// the n1 x n2 x n3 grid of Miller indices (taken modulo n) and transformed one axis at a time by
// direct DFTs with FP64-derived twiddles, in FP32 like the states the path stores.
//
// states_fused_kernel makes one state per CTA in shared memory, over the Miller indices that occur on each
// axis only (a sphere leaves most of the grid empty).  Measured at 20^3, 216 states: memset, scatter and
// three axis kernels took 105 us (global and L1 loads of every term, a modulo per output), now 41.
// Where its buffers do not fit a CTA (about 25^3 with every index used; 40^3 with a sphere half as
// wide as the grid), the axis kernels run; the sums and their order are the same.
#include <algorithm>
#include <cmath>

#include "gw_internal.cuh"

namespace gw {

namespace {

// C[b][idx[p]] = coef[b][p] (C zeroed beforehand); one block row per state.
__global__ void scatter_coef_kernel(const float2 *__restrict__ coef, int npw, const int *__restrict__ idx, int nr,
                                    float2 *__restrict__ C)
{
    const int b = blockIdx.y;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npw; p += gridDim.x * blockDim.x)
        C[(size_t)b * nr + idx[p]] = coef[(size_t)b * npw + p];
}

// out[b][..., j, ...] = scale sum_m in[b][..., m, ...] e^{+2 pi i m j / n} along the axis whose
// index has the given stride (n3 = 1, n2 = n3, n1 = n2 n3); tw[t] = e^{+2 pi i t / n}.
__global__ void dft_axis_kernel(const float2 *__restrict__ in, float2 *__restrict__ out, int nr, int n, int stride,
                                const float2 *__restrict__ tw, float scale)
{
    const int b = blockIdx.y;
    const float2 *x = in + (size_t)b * nr;
    float2 *y = out + (size_t)b * nr;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += gridDim.x * blockDim.x) {
        const int j = (r / stride) % n;
        const int base = r - j * stride;
        float ar = 0.f, ai = 0.f;
        int t = 0;
        for (int m = 0; m < n; ++m) {
            const float2 v = x[base + m * stride], w = tw[t];
            ar = fmaf(v.x, w.x, fmaf(-v.y, w.y, ar));
            ai = fmaf(v.x, w.y, fmaf(v.y, w.x, ai));
            t += j;
            if (t >= n)
                t -= n;
        }
        y[r] = make_float2(ar * scale, ai * scale);
    }
}

constexpr int SF_THREADS = 512;
constexpr int SF_JB = 8;  // outputs a thread makes of one line at a time
constexpr size_t SF_SMEM_MAX = 220 * 1024;

// Twiddle row of an axis: n values padded to whole blocks of outputs.
__host__ __device__ inline int sf_tw_pitch(int n) { return (n + SF_JB - 1) / SF_JB * SF_JB; }

// Shared memory, in float2, of a CTA that makes q3 of the n3 values j3: the twiddles, then two buffers.  The
// first holds the coefficients [m1][m2][m3 | 1], later [m1][n2][q3]; the second [m1][m2][q3 | 1] (odd
// pitches: the lanes of a warp are on different lines).
struct StateLayout {
    int tw[3], a, b, total;
    __host__ __device__ StateLayout(const StateAxes &x, int q3)
    {
        int o = 0;
        for (int i = 0; i < 3; ++i) {
            tw[i] = o;
            o += x.m[i] * sf_tw_pitch(i < 2 ? x.n[i] : q3);
        }
        a = o;
        const int c = x.m[0] * x.m[1] * (x.m[2] | 1), d = x.m[0] * x.n[1] * q3;
        o += c > d ? c : d;
        b = o;
        total = o + x.m[0] * x.m[1] * (q3 | 1);
    }
};

size_t sf_bytes(const StateAxes &ax, int parts)
{
    return StateLayout(ax, (ax.n[2] + parts - 1) / parts).total * sizeof(float2);
}

__device__ __forceinline__ int rank_of(unsigned long long mask, int i)  // used indices below i
{
    return __popcll(mask & ((1ull << i) - 1));
}

// acc[e] = sum_r x[r stride] tw[r pitch + e], e < JB, in the order of dft_axis_kernel.
template <int JB>
__device__ __forceinline__ void line_sums(const float2 *x, int stride, int m, const float2 *tw, int pitch, float2 *acc)
{
#pragma unroll
    for (int e = 0; e < JB; ++e)
        acc[e] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int r = 0; r < m; ++r) {
        const float2 v = x[r * stride];
        float4 w[JB / 2];
#pragma unroll
        for (int e = 0; e < JB / 2; ++e)
            w[e] = *reinterpret_cast<const float4 *>(tw + r * pitch + 2 * e);  // the same for every lane
#pragma unroll
        for (int e = 0; e < JB; ++e) {
            const float wx = e & 1 ? w[e / 2].z : w[e / 2].x, wy = e & 1 ? w[e / 2].w : w[e / 2].y;
            acc[e].x = fmaf(v.x, wx, fmaf(-v.y, wy, acc[e].x));
            acc[e].y = fmaf(v.x, wy, fmaf(v.y, wx, acc[e].y));
        }
    }
}

// One axis: lines x outputs j < n, a warp on 32 lines and a block of outputs at a time.  in(l) is the first
// value of line l (its values stride apart), out(l, j, value) stores.
template <class In, class Out>
__device__ __forceinline__ void axis_pass(int lines, int stride, int m, int n, const float2 *tw, In in, Out out)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, pitch = sf_tw_pitch(n);
    const int groups = (lines + 31) / 32, blocks = pitch / SF_JB;
    for (int t = warp; t < groups * blocks; t += SF_THREADS / 32) {
        const int g = t / blocks, j0 = (t - g * blocks) * SF_JB, l = g * 32 + lane;
        if (l >= lines)
            continue;
        const float2 *x = in(l);
        float2 acc[SF_JB];
        if (n - j0 <= SF_JB / 2)
            line_sums<SF_JB / 2>(x, stride, m, tw + j0, pitch, acc);
        else
            line_sums<SF_JB>(x, stride, m, tw + j0, pitch, acc);
#pragma unroll
        for (int e = 0; e < SF_JB; ++e)
            if (j0 + e < n)
                out(l, j0 + e, acc[e]);
    }
}

// A state, or the half of it with blockIdx.y's values j3, per CTA.  Every step is bound by shared memory and FMAs about equally: a thread reads one value
// and eight twiddles (broadcast) for 32 FMAs.
__global__ void __launch_bounds__(SF_THREADS) states_fused_kernel(const float2 *__restrict__ coef, int npw,
                                                                  const int *__restrict__ idx, StateAxes ax,
                                                                  const float2 *__restrict__ tw, float scale,
                                                                  float2 *__restrict__ out)
{
    extern __shared__ __align__(16) float2 sf_smem[];
    __shared__ int used[3][64];
    const int tid = threadIdx.x, n2 = ax.n[1], n3 = ax.n[2], m1 = ax.m[0], m2 = ax.m[1], m3 = ax.m[2];
    const int qmax = (n3 + gridDim.y - 1) / gridDim.y, j30 = blockIdx.y * qmax, q3 = min(qmax, n3 - j30);
    const StateLayout L(ax, qmax);
    float2 *A = sf_smem + L.a, *B = sf_smem + L.b;
    if (tid < 192) {
        const int a = tid >> 6, i = tid & 63;
        if (ax.mask[a] >> i & 1)
            used[a][rank_of(ax.mask[a], i)] = i;
    }
    const int pc = m3 | 1, pb = q3 | 1;
    for (int t = tid; t < m1 * m2 * pc; t += SF_THREADS)
        A[t] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int a = 0, o = 0; a < 3; o += ax.n[a], ++a) {
        const int n = ax.n[a], jn = a < 2 ? n : q3, j0 = a < 2 ? 0 : j30, pitch = sf_tw_pitch(jn);
        for (int t = tid; t < ax.m[a] * pitch; t += SF_THREADS) {
            const int r = t / pitch, j = t - r * pitch;
            sf_smem[L.tw[a] + t] = j < jn ? tw[o + used[a][r] * (j0 + j) % n] : make_float2(0.f, 0.f);
        }
    }
    const float2 *src = coef + (size_t)blockIdx.x * npw;
    for (int p = tid; p < npw; p += SF_THREADS) {
        const int lin = idx[p], q = lin / n3, i3 = lin - q * n3, i1 = q / n2, i2 = q - i1 * n2;
        A[(rank_of(ax.mask[0], i1) * m2 + rank_of(ax.mask[1], i2)) * pc + rank_of(ax.mask[2], i3)] = src[p];
    }
    __syncthreads();
    axis_pass(m1 * m2, 1, m3, q3, sf_smem + L.tw[2], [&](int l) { return A + l * pc; },
              [&](int l, int j, float2 v) { B[l * pb + j] = v; });
    __syncthreads();
    axis_pass(m1 * q3, pb, m2, n2, sf_smem + L.tw[1],
              [&](int l) {
                  const int r1 = l / q3;
                  return B + r1 * m2 * pb + l - r1 * q3;
              },
              [&](int l, int j, float2 v) {
                  const int r1 = l / q3;
                  A[(r1 * n2 + j) * q3 + l - r1 * q3] = v;
              });
    __syncthreads();
    float2 *y = out + (size_t)blockIdx.x * ax.n[0] * n2 * n3 + j30;
    axis_pass(n2 * q3, n2 * q3, m1, ax.n[0], sf_smem + L.tw[0], [&](int l) { return A + l; },
              [&](int l, int j, float2 v) {
                  const int j2 = l / q3;
                  y[((size_t)j * n2 + j2) * n3 + l - j2 * q3] = make_float2(v.x * scale, v.y * scale);
              });
}

// P~ of one k-point into the running sum of Sec. 4.1's (1/N_k) sum over k:
// PG = (acc ? sum : 0) + w PG, in FP32 like P~ itself.
__global__ void kweight_kernel(float2 *__restrict__ PG, const float2 *__restrict__ sum, size_t n, float w, int acc)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float2 v = PG[i];
        v.x *= w;
        v.y *= w;
        if (acc) {
            v.x += sum[i].x;
            v.y += sum[i].y;
        }
        PG[i] = v;
    }
}

}  // namespace

cudaError_t launch_kweight(float2 *PG, const float2 *sum, size_t n, float w, bool acc, cudaStream_t s)
{
    const int grid = static_cast<int>(std::min<size_t>((n + 255) / 256, 152 * 8));
    kweight_kernel<<<std::max(1, grid), 256, 0, s>>>(PG, sum, n, w, acc ? 1 : 0);
    count_launches(1);
    return cudaGetLastError();
}

bool states_fused(const StateAxes &ax)
{
    return sf_bytes(ax, 1) <= SF_SMEM_MAX;
}

// coef: [nb][npw] complex64 (device); idx: [npw] linear grid index of each Miller index (device);
// tw: [n1 | n2 | n3] twiddle tables (device); work: nb * nr complex64 (unused where states_fused(ax));
// out: [nb][nr] complex64.
cudaError_t launch_states_from_g(const float2 *coef, int nb, int npw, const int *idx, const StateAxes &ax,
                                 const float2 *tw, float2 *work, float2 *out, cudaStream_t s)
{
    const int n1 = ax.n[0], n2 = ax.n[1], n3 = ax.n[2], nr = n1 * n2 * n3;
    const float scale = static_cast<float>(1.0 / std::sqrt(static_cast<double>(nr)));
    if (states_fused(ax)) {
        // halves where they let two CTAs share an SM and whole states do not: 20^3 and 216 states, two k-points
        // of a sum 875 -> 861 us (216 whole states are 1.4 waves of one CTA per SM)
        const int parts = ax.n[2] > 1 && sf_bytes(ax, 1) > SF_SMEM_MAX / 2 && sf_bytes(ax, 2) <= SF_SMEM_MAX / 2 ? 2 : 1;
        const size_t smem = sf_bytes(ax, parts);
        const cudaError_t e =
            cudaFuncSetAttribute(states_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        states_fused_kernel<<<dim3(nb, parts), SF_THREADS, smem, s>>>(coef, npw, idx, ax, tw, scale, out);
        count_launches(1);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(work, 0, (size_t)nb * nr * sizeof(float2), s);
    if (e != cudaSuccess)
        return e;
    for (int b0 = 0; b0 < nb; b0 += 65535) {  // grid y is one state per row, at most 65535
        const int nbb = std::min(65535, nb - b0);
        const size_t off = (size_t)b0 * nr;
        const dim3 gs((npw + 255) / 256, nbb);
        scatter_coef_kernel<<<gs, 256, 0, s>>>(coef + (size_t)b0 * npw, npw, idx, nr, work + off);
        const dim3 g((nr + 255) / 256, nbb);
        dft_axis_kernel<<<g, 256, 0, s>>>(work + off, out + off, nr, n3, 1, tw + n1 + n2, 1.0f);   // m3 -> j3
        dft_axis_kernel<<<g, 256, 0, s>>>(out + off, work + off, nr, n2, n3, tw + n1, 1.0f);       // m2 -> j2
        dft_axis_kernel<<<g, 256, 0, s>>>(work + off, out + off, nr, n1, n2 * n3, tw, scale);      // m1 -> j1
        count_launches(4);
    }
    return cudaGetLastError();
}

}  // namespace gw
