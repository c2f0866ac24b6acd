// Element-wise and reduction kernels of the surrogate network (the GEMMs are
// in sur_gemm.cu).  All arithmetic in FP32; BF16 copies feed the GEMMs.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "sur_adam.cuh"
#include "sur_internal.h"

namespace es {
namespace {

inline int blocks_for(size_t n, int t = 256)
{
    size_t b = (n + t - 1) / t;
    return (int)(b > 65535 * 8 ? 65535 * 8 : b);
}

__global__ void scale_kernel(float* C, int M, int N, int ldc, float s)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)M * N; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / N, c = i % N;
        C[r * ldc + c] = s == 0.f ? 0.f : C[r * ldc + c] * s;  // s = 0 also clears NaN
    }
}

__global__ void cast_kernel(const float* x, __nv_bfloat16* y, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16(x[i]);
}

// one thread per sine and cosine pair of a position, and one for its three coordinates and the padding
__global__ void features_kernel(const float* pos, int B, int nfreq, int width, __nv_bfloat16* X)
{
    const int per = 3 * nfreq + 1, i = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = i / per, q = i - b * per;
    if (b >= B) return;
    __nv_bfloat16* row = X + (size_t)b * width;
    if (q < 3 * nfreq) {
        float s, c;
        sincospif(ldexpf(pos[3 * b + q % 3], q / 3), &s, &c);  // sin, cos of 2^j pi p
        row[3 + 2 * q] = __float2bfloat16(s);
        row[4 + 2 * q] = __float2bfloat16(c);
    } else {
        for (int a = 0; a < 3; ++a) row[a] = __float2bfloat16(pos[3 * b + a]);
        for (int k = 3 + 6 * nfreq; k < width; ++k) row[k] = __float2bfloat16(0.f);
    }
}

__global__ void contract_kernel(const float* M6, const float* dZ, int B, int K, float* dA, __nv_bfloat16* dAb)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)B * K; i += (size_t)gridDim.x * blockDim.x) {
        const size_t b = i / K, k = i % K;
        float s = 0.f;
        for (int c = 0; c < 6; ++c) s += M6[6 * b + c] * dZ[b * 6 * K + (size_t)c * K + k];
        dA[i] = s;
        dAb[i] = __float2bfloat16(s);
    }
}

// Loss in component-scaled units: with y = s_c u and tau = t / s_c,
// l_b = sum_c |u_c - tau_c|^2 / (sum_c |tau_c|^2 + eps) -- the relative L2
// error (squared) of the whole 4C seismogram after each component is divided
// by its scale.  Pass 1 (one block per sample and component) forms the two sums
// of each, in a fixed order, so that two calls see the same dL/du to the last
// bit of its BF16 rounding.
__global__ void loss_sums_kernel(const float* U, const float* T, const float* scale, long long Dc, float2* acc)
{
    const int b = blockIdx.x, c = blockIdx.y;
    const size_t base = ((size_t)b * 4 + c) * Dc;
    const float inv = 1.f / scale[c];
    float se = 0.f, st = 0.f;
    for (long long i = threadIdx.x; i < Dc; i += blockDim.x) {
        const float tau = T[base + i] * inv;
        const float d = U[base + i] - tau;
        se += d * d;
        st += tau * tau;
    }
    for (int o = 16; o > 0; o >>= 1) {
        se += __shfl_down_sync(0xffffffffu, se, o);
        st += __shfl_down_sync(0xffffffffu, st, o);
    }
    __shared__ float2 part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_float2(se, st);
    __syncthreads();
    if (threadIdx.x == 0) {
        float2 sum = part[0];
        for (int i = 1; i < 8; ++i) {
            sum.x += part[i].x;
            sum.y += part[i].y;
        }
        acc[4 * b + c] = sum;
    }
}

// Pass 2 on tiles of 64 samples x 64 columns: dL/du in BF16 both row-major and
// transposed (the K-major operand of the decoder's gradient), the second through a
// shared [column][sample] tile; the first column tile also writes the losses.
// What bounds it is HBM.  256 x 262144 (one GB300): 120 us, 164 with two-byte
// stores and 136 more for a transpose kernel that read them back.
constexpr int LT = 64, LT_LD = LT + 2;
__global__ void __launch_bounds__(256) loss_grad_kernel(const float* U, const float* T, const float* scale, int B,
                                                        long long Dc, float eps, const float2* acc, __nv_bfloat16* dU,
                                                        __nv_bfloat16* dUT, float* loss, float* per_sample, bool vec,
                                                        int nx)
{
    __shared__ __align__(16) __nv_bfloat16 tt[LT][LT_LD];
    __shared__ float g[LT];
    // column tiles fastest, in one dimension (any number of samples)
    const int tx = blockIdx.x % nx;
    const long long D = 4 * Dc, d0 = (long long)tx * LT;
    const int b0 = (int)(blockIdx.x / nx) * LT;
    if (threadIdx.x < LT && b0 + (int)threadIdx.x < B) {
        const int b = b0 + threadIdx.x;
        const float2 a0 = acc[4 * b], a1 = acc[4 * b + 1], a2 = acc[4 * b + 2], a3 = acc[4 * b + 3];
        const float den = a0.y + a1.y + a2.y + a3.y + eps;
        g[threadIdx.x] = 2.f / ((float)B * den);
        if (tx == 0) {
            const float lb = (a0.x + a1.x + a2.x + a3.x) / den;
            if (per_sample) per_sample[b] = lb;
            atomicAdd(loss, lb / B);
        }
    }
    if (!dU) return;
    __syncthreads();
    const int q = threadIdx.x & 15, r = threadIdx.x >> 4;  // 16 column quads x 16 samples per sweep
    const long long d = d0 + 4 * q;
    if (d < D) {  // Dc is a multiple of 8: a quad lies within one component
        const float inv = 1.f / scale[d / Dc];
#pragma unroll
        for (int i = r; i < LT; i += 16) {
            if (b0 + i >= B) break;
            const size_t at = (size_t)(b0 + i) * D + d;
            const float4 u = *reinterpret_cast<const float4*>(U + at);
            const float4 t = vec ? *reinterpret_cast<const float4*>(T + at)
                                 : make_float4(T[at], T[at + 1], T[at + 2], T[at + 3]);
            const float4 v = make_float4(g[i] * (u.x - t.x * inv), g[i] * (u.y - t.y * inv), g[i] * (u.z - t.z * inv),
                                         g[i] * (u.w - t.w * inv));
            const uint2 w = pack_bf16x4(v);
            *reinterpret_cast<uint2*>(dU + at) = w;
            const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&w);
#pragma unroll
            for (int k = 0; k < 4; ++k) tt[4 * q + k][i] = e[k];
        }
    }
    __syncthreads();
    for (int j = r; j < LT; j += 16) {  // four samples of column d0 + j (B is a multiple of 8)
        if (d0 + j >= D || b0 + 4 * q >= B) continue;
        const uint32_t* w = reinterpret_cast<const uint32_t*>(&tt[j][4 * q]);
        *reinterpret_cast<uint2*>(dUT + (size_t)(d0 + j) * B + b0 + 4 * q) = make_uint2(w[0], w[1]);
    }
}

// x ~ N(0, std^2) from a counter-based hash (splitmix64 of seed + index) and Box-Muller
__global__ void init_normal_kernel(float* p, size_t n, float std, unsigned long long seed)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const float u1 = ((z >> 40) + 1) * (1.0f / 16777217.0f);
        const float u2 = ((z >> 16) & 0xFFFFFF) * (1.0f / 16777216.0f);
        p[i] = std * sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
    }
}

// ss[c] += sum of t^2 over component c of every sample ([n][4][Dc])
__global__ void comp_sumsq_kernel(const float* T, int n, long long Dc, float* ss)
{
    const int b = blockIdx.x, c = blockIdx.y;
    const float* t = T + ((size_t)b * 4 + c) * Dc;
    float s = 0.f;
    for (long long i = threadIdx.x; i < Dc; i += blockDim.x) s += t[i] * t[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(ss + c, s);
}

// out[b][d] = sum_c mt[b][c] G[loc[b]][c][d]
__global__ void combine_kernel(const float* G, long long D, const int* loc, const float* mt, int B, float* out)
{
    const int b = blockIdx.y;
    const float* g = G + (size_t)loc[b] * 6 * D;
    const float m0 = mt[6 * b], m1 = mt[6 * b + 1], m2 = mt[6 * b + 2], m3 = mt[6 * b + 3], m4 = mt[6 * b + 4],
                m5 = mt[6 * b + 5];
    for (long long d = blockIdx.x * (long long)blockDim.x + threadIdx.x; d < D; d += (long long)gridDim.x * blockDim.x)
        out[(size_t)b * D + d] = m0 * g[d] + m1 * g[D + d] + m2 * g[2 * D + d] + m3 * g[3 * D + d] + m4 * g[4 * D + d] +
                                 m5 * g[5 * D + d];
}

// 32 columns per block; warp w sums rows w, w + 8, ... in order, then the warps' sums are added in order
__global__ void colsum_kernel(const float* G, int B, int N, float* db)
{
    __shared__ float part[8][32];
    const int n = blockIdx.x * 32 + threadIdx.x % 32, w = threadIdx.x / 32;
    float s = 0.f;
    if (n < N)
#pragma unroll 8
        for (int b = w; b < B; b += 8) s += G[(size_t)b * N + n];
    part[w][threadIdx.x % 32] = s;
    __syncthreads();
    if (w > 0 || n >= N) return;
    for (int i = 1; i < 8; ++i) s += part[i][threadIdx.x];
    db[n] = s;
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2, __nv_bfloat16* pb)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float pi = p[i], mi = m[i], vi = v[i];
        adam_one(pi, g[i], mi, vi, lr, b1, b2, eps, c1, c2);
        m[i] = mi;
        v[i] = vi;
        p[i] = pi;
        if (pb) pb[i] = __float2bfloat16(pi);
    }
}

// four parameters per thread and iteration (n4 groups of four, 16-byte aligned)
__global__ void adam4_kernel(float4* p, const float4* g, float4* m, float4* v, size_t n4,
                             const AdamStep w, uint2* pb)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 pi = p[i], mi = m[i], vi = v[i];
        adam_four(pi, g[i], mi, vi, w);
        m[i] = mi;
        v[i] = vi;
        p[i] = pi;
        if (pb) pb[i] = pack_bf16x4(pi);
    }
}

// The step on 64 x 64 tiles of a row-major [rows][cols] block: the update and the row-major BF16 copy four
// columns per thread, the transposed copy through a shared [column][row] tile, four rows per thread.  HBM
// bounds it: 4608 x 262144 (one GB300) 5.7 ms, 32 bytes a weight at 6.8 TB/s.
constexpr int AT = 64, AT_LD = AT + 4;
__global__ void __launch_bounds__(256) adam_t_kernel(float* p, const float* g, float* m, float* v, long long rows,
                                                     long long cols, const AdamStep w, __nv_bfloat16* pb, __nv_bfloat16* pt)
{
    __shared__ __align__(16) __nv_bfloat16 tt[AT][AT_LD];
    const long long c0 = (long long)blockIdx.x * AT, r0 = (long long)blockIdx.y * AT;
    const int cq = threadIdx.x & 15, rq = threadIdx.x >> 4;  // 16 column quads x 16 rows per sweep
    for (int i = rq; i < AT; i += 16) {
        const long long r = r0 + i, c = c0 + 4 * cq;
        if (r >= rows || c >= cols) continue;
        const size_t k = (size_t)r * cols + c;
        float4 pi = *reinterpret_cast<const float4*>(p + k);
        float4 mi = *reinterpret_cast<const float4*>(m + k), vi = *reinterpret_cast<const float4*>(v + k);
        adam_four(pi, *reinterpret_cast<const float4*>(g + k), mi, vi, w);
        *reinterpret_cast<float4*>(m + k) = mi;
        *reinterpret_cast<float4*>(v + k) = vi;
        *reinterpret_cast<float4*>(p + k) = pi;
        const uint2 q = pack_bf16x4(pi);
        *reinterpret_cast<uint2*>(pb + k) = q;
        const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&q);
#pragma unroll
        for (int j = 0; j < 4; ++j) tt[4 * cq + j][i] = e[j];
    }
    __syncthreads();
    for (int j = rq; j < AT; j += 16) {
        const long long c = c0 + j, r = r0 + 4 * cq;
        if (c < cols && r < rows) *reinterpret_cast<uint2*>(pt + (size_t)c * rows + r) = *reinterpret_cast<const uint2*>(&tt[j][4 * cq]);
    }
}

}  // namespace

cudaError_t scale_f32(float* C, int M, int N, int ldc, float s, cudaStream_t st)
{
    scale_kernel<<<blocks_for((size_t)M * N), 256, 0, st>>>(C, M, N, ldc, s);
    return cudaGetLastError();
}

// 64 x 64 tiles through shared memory (row padded by 2 elements: the column
// reads of the second half hit 32 distinct banks)
__global__ void transpose_bf16_kernel(const __nv_bfloat16* __restrict__ in, long long rows, long long cols,
                                      __nv_bfloat16* __restrict__ out)
{
    __shared__ __nv_bfloat16 t[64][66];
    const long long c0 = (long long)blockIdx.x * 64, r0 = (long long)blockIdx.y * 64;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int i = ty; i < 64; i += 8)
        for (int j = tx; j < 64; j += 32) {
            const long long r = r0 + i, c = c0 + j;
            t[i][j] = (r < rows && c < cols) ? in[r * cols + c] : __float2bfloat16(0.f);
        }
    __syncthreads();
    for (int i = ty; i < 64; i += 8)
        for (int j = tx; j < 64; j += 32) {
            const long long c = c0 + i, r = r0 + j;
            if (c < cols && r < rows) out[c * rows + r] = t[j][i];
        }
}

cudaError_t transpose_bf16(const __nv_bfloat16* in, long long rows, long long cols, __nv_bfloat16* out,
                           cudaStream_t st)
{
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    const long long gx = (cols + 63) / 64, gy = (rows + 63) / 64;
    if (gx > 0x7fffffffLL || gy > 65535) return cudaErrorInvalidValue;
    transpose_bf16_kernel<<<dim3((unsigned)gx, (unsigned)gy), 256, 0, st>>>(in, rows, cols, out);
    return cudaGetLastError();
}

cudaError_t cast_bf16(const float* x, __nv_bfloat16* y, size_t n, cudaStream_t st)
{
    cast_kernel<<<blocks_for(n), 256, 0, st>>>(x, y, n);
    return cudaGetLastError();
}

cudaError_t sur_features(const float* pos, int B, int nfreq, int width, __nv_bfloat16* X, cudaStream_t st)
{
    if (3 + 6 * nfreq > width) return cudaErrorInvalidValue;
    features_kernel<<<(B * (3 * nfreq + 1) + 127) / 128, 128, 0, st>>>(pos, B, nfreq, width, X);
    return cudaGetLastError();
}

cudaError_t sur_contract(const float* M6, const float* dZ, int B, int K, float* dA, __nv_bfloat16* dAb, cudaStream_t st)
{
    contract_kernel<<<blocks_for((size_t)B * K), 256, 0, st>>>(M6, dZ, B, K, dA, dAb);
    return cudaGetLastError();
}

cudaError_t sur_loss(const float* U, const float* T, const float* scale, int B, long long Dc, float eps,
                     __nv_bfloat16* dU, __nv_bfloat16* dUT, float* loss, float* acc, float* per_sample, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(float), st);
    if (e != cudaSuccess) return e;
    float2* sums = reinterpret_cast<float2*>(acc);
    loss_sums_kernel<<<dim3(B, 4), 256, 0, st>>>(U, T, scale, Dc, sums);
    const long long nx = dU ? (4 * Dc + LT - 1) / LT : 1;
    const long long tiles = nx * ((B + LT - 1) / LT);
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    loss_grad_kernel<<<(unsigned)tiles, 256, 0, st>>>(U, T, scale, B, Dc, eps, sums, dU, dUT, loss, per_sample,
                                                     (reinterpret_cast<uintptr_t>(T) & 15) == 0, (int)nx);
    return cudaGetLastError();
}

cudaError_t sur_init_normal(float* p, size_t n, float std, unsigned long long seed, cudaStream_t st)
{
    init_normal_kernel<<<blocks_for(n), 256, 0, st>>>(p, n, std, seed);
    return cudaGetLastError();
}

cudaError_t sur_comp_sumsq(const float* T, int n, long long Dc, float* ss, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(ss, 0, 4 * sizeof(float), st);
    if (e != cudaSuccess) return e;
    comp_sumsq_kernel<<<dim3(n, 4), 256, 0, st>>>(T, n, Dc, ss);
    return cudaGetLastError();
}

cudaError_t sur_combine(const float* G, long long D, const int* loc, const float* mt, int B, float* out,
                        cudaStream_t st)
{
    const long long nb = std::min<long long>((D + 255) / 256, 1024);
    combine_kernel<<<dim3((unsigned)nb, B), 256, 0, st>>>(G, D, loc, mt, B, out);
    return cudaGetLastError();
}

cudaError_t sur_colsum(const float* G, int B, int N, float* db, cudaStream_t st)
{
    colsum_kernel<<<(N + 31) / 32, 256, 0, st>>>(G, B, N, db);
    return cudaGetLastError();
}

cudaError_t sur_adam(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2, float eps,
                     int t, __nv_bfloat16* pb, cudaStream_t st)
{
    const AdamStep w = adam_step(lr, b1, b2, eps, t);
    const uintptr_t al = reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) |
                         reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v);
    if (n % 4 == 0 && (al & 15) == 0 && (reinterpret_cast<uintptr_t>(pb) & 7) == 0) {
        adam4_kernel<<<blocks_for(n / 4), 256, 0, st>>>(
            reinterpret_cast<float4*>(p), reinterpret_cast<const float4*>(g), reinterpret_cast<float4*>(m),
            reinterpret_cast<float4*>(v), n / 4, w,
            reinterpret_cast<uint2*>(pb));
    } else {
        adam_kernel<<<blocks_for(n), 256, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, w.c1, w.c2, pb);
    }
    return cudaGetLastError();
}

cudaError_t sur_adam_t(float* p, const float* g, float* m, float* v, long long rows, long long cols, float lr, float b1,
                       float b2, float eps, int t, __nv_bfloat16* pb, __nv_bfloat16* pt, cudaStream_t st)
{
    const long long gx = (cols + AT - 1) / AT, gy = (rows + AT - 1) / AT;
    if (rows % 4 || cols % 4 || gx > 0x7fffffffLL || gy > 65535) return cudaErrorInvalidValue;
    adam_t_kernel<<<dim3((unsigned)gx, (unsigned)gy), 256, 0, st>>>(p, g, m, v, rows, cols, adam_step(lr, b1, b2, eps, t), pb,
                                                                   pt);
    return cudaGetLastError();
}

}  // namespace es
