// BF16-input, FP32-accumulate GEMM for the surrogate network:
//   C[M][N] = alpha * op(A)[M][K] op(B)[K][N] + beta * C
// A is row-major [M][K] (lda) or, with a_t, stored [K][M]; B is stored
// [N][K] (b_nk, "column-major") or [K][N].  C is FP32 row-major (ldc).
// With split_k > 1 the K range is cut into slices whose partial products are
// added into C with atomics (C must hold beta * C already; alpha applies).
//
// CTA tile 128 x 128 x 32, 8 warps (2 x 4), warp tile 64 x 32, tensor-core
// mma.sync m16n8k16 bf16 -> f32; operand fragments come from shared memory
// through ldmatrix (transposing on the fly for the [K][M] / [K][N] storage
// orders); global -> shared tiles move with 16-byte cp.async, double
// buffered.  Out-of-range rows and columns are zero-filled.
// The K-major order of both operands (A [M][K], B [N][K]) runs on the
// tcgen05 tensor cores instead (sur_gemm_tc.cu).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sur_internal.h"

namespace es {
namespace {

constexpr int BM = 128, BN = 128, BK = 32, PAD = 8;
constexpr int THREADS = 256;

__device__ __forceinline__ void cp16(void* dst, const void* src, bool ok)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(K) : "memory"); }

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void* p)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}
__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void* p)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// shared tiles: A as [BM][BK+PAD] (k contiguous) or [BK][BM+PAD]; B as
// [BN][BK+PAD] or [BK][BN+PAD]
template <bool AT, bool BNK>
struct Smem {
    static constexpr int A_ELEMS = AT ? BK * (BM + PAD) : BM * (BK + PAD);
    static constexpr int B_ELEMS = BNK ? BN * (BK + PAD) : BK * (BN + PAD);
    __nv_bfloat16 a[2][A_ELEMS];
    __nv_bfloat16 b[2][B_ELEMS];
};

template <bool AT, bool BNK>
__global__ void __launch_bounds__(THREADS) gemm_bf16_kernel(int M, int N, int K, const __nv_bfloat16* __restrict__ A,
                                                           int lda, const __nv_bfloat16* __restrict__ B, int ldb,
                                                           float* __restrict__ C, int ldc, float alpha, float beta,
                                                           int k_per_split)
{
    __shared__ __align__(128) Smem<AT, BNK> sm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 2, wn = warp & 3;  // warp tile 64 x 32
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int kbeg = blockIdx.z * k_per_split;
    const int kend = min(K, kbeg + k_per_split);
    const int ntiles = (kend - kbeg + BK - 1) / BK;

    auto load_tile = [&](int stage, int k0) {
        // A: 512 chunks of 8 bf16
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c = tid + i * THREADS;
            if (!AT) {
                const int r = c >> 2, kc = (c & 3) * 8;  // row m, 4 chunks per row
                const int gm = m0 + r, gk = k0 + kc;
                const bool ok = gm < M && gk < kend;
                cp16(&sm.a[stage][r * (BK + PAD) + kc], A + (ok ? (size_t)gm * lda + gk : 0), ok);
            } else {
                const int r = c >> 4, mc = (c & 15) * 8;  // row k, 16 chunks per row
                const int gk = k0 + r, gm = m0 + mc;
                const bool ok = gk < kend && gm < M;
                cp16(&sm.a[stage][r * (BM + PAD) + mc], A + (ok ? (size_t)gk * lda + gm : 0), ok);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c = tid + i * THREADS;
            if (BNK) {
                const int r = c >> 2, kc = (c & 3) * 8;
                const int gn = n0 + r, gk = k0 + kc;
                const bool ok = gn < N && gk < kend;
                cp16(&sm.b[stage][r * (BK + PAD) + kc], B + (ok ? (size_t)gn * ldb + gk : 0), ok);
            } else {
                const int r = c >> 4, nc = (c & 15) * 8;
                const int gk = k0 + r, gn = n0 + nc;
                const bool ok = gk < kend && gn < N;
                cp16(&sm.b[stage][r * (BN + PAD) + nc], B + (ok ? (size_t)gk * ldb + gn : 0), ok);
            }
        }
        cp_commit();
    };

    float acc[4][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;

    if (ntiles > 0) load_tile(0, kbeg);
    for (int t = 0; t < ntiles; ++t) {
        const int st = t & 1;
        if (t + 1 < ntiles) {
            load_tile(st ^ 1, kbeg + (t + 1) * BK);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            unsigned af[4][4], bf[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int mb = wm * 64 + i * 16;
                if (!AT) {
                    const __nv_bfloat16* p = &sm.a[st][(mb + (lane & 15)) * (BK + PAD) + kk + (lane >> 4) * 8];
                    ldsm_x4(af[i], p);
                } else {
                    const int k = kk + (lane & 7) + ((lane >> 4) << 3);
                    const int m = mb + (((lane >> 3) & 1) << 3);
                    ldsm_x4_t(af[i], &sm.a[st][k * (BM + PAD) + m]);
                }
            }
#pragma unroll
            for (int j = 0; j < 4; j += 2) {  // two n8 tiles per ldmatrix.x4
                const int nb = wn * 32 + j * 8;
                unsigned r[4];
                if (BNK) {
                    // matrices: (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15)
                    const int n = nb + (lane & 7) + ((lane >> 4) << 3);
                    const int k = kk + (((lane >> 3) & 1) << 3);
                    ldsm_x4(r, &sm.b[st][n * (BK + PAD) + k]);
                } else {
                    // stored [k][n]: same four matrices, transposed on load
                    const int k = kk + (lane & 7) + (((lane >> 3) & 1) << 3);
                    const int n = nb + ((lane >> 4) << 3);
                    ldsm_x4_t(r, &sm.b[st][k * (BN + PAD) + n]);
                }
                bf[j][0] = r[0];
                bf[j][1] = r[1];
                bf[j + 1][0] = r[2];
                bf[j + 1][1] = r[3];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma16816(acc[i][j], af[i], bf[j][0], bf[j][1]);
        }
        __syncthreads();
    }

    // accumulator element e of tile (i, j): row = lane/4 (+8 for e >= 2), col = 2 (lane % 4) + (e & 1)
    const bool split = gridDim.z > 1;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int r = m0 + wm * 64 + i * 16 + (lane >> 2) + ((e >> 1) << 3);
                const int c = n0 + wn * 32 + j * 8 + ((lane & 3) << 1) + (e & 1);
                if (r < M && c < N) {
                    float* out = C + (size_t)r * ldc + c;
                    const float v = alpha * acc[i][j][e];
                    if (split) atomicAdd(out, v);
                    else *out = beta == 0.f ? v : v + beta * *out;
                }
            }
}

// ---------------------------------------------------------------------------
// The layers of the encoder: products of a batch with weights of a few hundred
// rows, far too small to fill the device in 128 x 128 tiles.  CTA tile 32 x 64, 4
// warps (2 x 2, 16 x 32 each), k-slabs of 64 through a ring of five, so that
// what bounds it is the latency of one slab per five, and the elementwise step
// that follows a layer in its epilogue (MlpEpilogue).
// 256 x 768 x 768 (one GB300): 8.8 us with bias, ReLU and the BF16 copy, 20.6 + 3.3
// in 12 CTAs of the general kernel and one of its own; its backward products 6.2
// against 11.2 (weights) and 9.4 against 14.6 + 3.8 (tcgen05, 6 CTAs; rows).  A
// training step of a small network (hidden layers of 128, decoder 96 x 256) falls
// from 218 to 149 us, a serving batch of 1024 at full size from 1.82 to 1.78 ms.
// Products with many tiles go to the general kernels and a pass of their own for
// the elementwise step (small_layer).
constexpr int LM = 32, LN = 64, LK = 64, LS = 5, LTHREADS = 128;

template <bool AT, bool BNK>
struct LayerTile {
    static constexpr int LDA = AT ? LM + PAD : LK + PAD, LDB = BNK ? LK + PAD : LN + PAD;
    static constexpr int A = (AT ? LK : LM) * LDA, B = (BNK ? LN : LK) * LDB;
    static constexpr int BYTES = LS * (A + B) * 2;
};

template <bool AT, bool BNK>
__global__ void __launch_bounds__(LTHREADS)
layer_kernel(int M, int N, int K, const __nv_bfloat16* __restrict__ A, int lda, const __nv_bfloat16* __restrict__ B,
             int ldb, float* __restrict__ C, const MlpEpilogue ep)
{
    using L = LayerTile<AT, BNK>;
    extern __shared__ __align__(128) __nv_bfloat16 ring[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    const int ntn = (N + LN - 1) / LN;  // tiles in a row of them; rows in one dimension, which takes any batch
    const int m0 = (int)(blockIdx.x / ntn) * LM, n0 = (int)(blockIdx.x % ntn) * LN;
    const int nk = (K + LK - 1) / LK;

    auto load = [&](int t) {
        if (t < nk) {
            __nv_bfloat16* a = ring + t % LS * (L::A + L::B);
            __nv_bfloat16* b = a + L::A;
            const int k0 = t * LK;
#pragma unroll
            for (int i = 0; i < LM * LK / 8 / LTHREADS; ++i) {
                const int c = tid + i * LTHREADS;
                const int r = AT ? c / (LM / 8) : c / (LK / 8), q = AT ? c % (LM / 8) * 8 : c % (LK / 8) * 8;
                const int gk = k0 + (AT ? r : q), gm = m0 + (AT ? q : r);
                const bool ok = gk < K && gm < M;
                cp16(a + r * L::LDA + q, A + (ok ? (AT ? (size_t)gk * lda + gm : (size_t)gm * lda + gk) : 0), ok);
            }
#pragma unroll
            for (int i = 0; i < LN * LK / 8 / LTHREADS; ++i) {
                const int c = tid + i * LTHREADS, r = c / 8, q = c % 8 * 8;  // LN == LK: 8 chunks a row
                const int gk = k0 + (BNK ? q : r), gn = n0 + (BNK ? r : q);
                const bool ok = gk < K && gn < N;
                cp16(b + r * L::LDB + q, B + (ok ? (BNK ? (size_t)gn * ldb + gk : (size_t)gk * ldb + gn) : 0), ok);
            }
        }
        cp_commit();  // an empty group past the end keeps the count
    };

    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
#pragma unroll
    for (int t = 0; t < LS - 1; ++t) load(t);
    for (int t = 0; t < nk; ++t) {
        cp_wait<LS - 2>();
        __syncthreads();  // slab t is there, slab t - 1 has been read
        load(t + LS - 1);
        const __nv_bfloat16* a = ring + t % LS * (L::A + L::B);
        const __nv_bfloat16* b = a + L::A;
#pragma unroll
        for (int kk = 0; kk < LK; kk += 16) {
            unsigned af[4], bf[4][2];
            if (!AT) {
                ldsm_x4(af, a + (wm * 16 + (lane & 15)) * L::LDA + kk + (lane >> 4) * 8);
            } else {
                const int k = kk + (lane & 7) + ((lane >> 4) << 3), m = wm * 16 + (((lane >> 3) & 1) << 3);
                ldsm_x4_t(af, a + k * L::LDA + m);
            }
#pragma unroll
            for (int j = 0; j < 4; j += 2) {  // two n8 tiles per ldmatrix.x4 (see gemm_bf16_kernel)
                const int nb = wn * 32 + j * 8;
                unsigned r[4];
                if (BNK) {
                    const int n = nb + (lane & 7) + ((lane >> 4) << 3), k = kk + (((lane >> 3) & 1) << 3);
                    ldsm_x4(r, b + n * L::LDB + k);
                } else {
                    const int k = kk + (lane & 7) + (((lane >> 3) & 1) << 3), n = nb + ((lane >> 4) << 3);
                    ldsm_x4_t(r, b + k * L::LDB + n);
                }
                bf[j][0] = r[0];
                bf[j][1] = r[1];
                bf[j + 1][0] = r[2];
                bf[j + 1][1] = r[3];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) mma16816(acc[j], af, bf[j][0], bf[j][1]);
        }
    }

    // pairs of columns (N is a multiple of 8): rows lane / 4 and + 8, columns 2 (lane % 4) of each n8 tile
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = m0 + wm * 16 + (lane >> 2) + 8 * h, c = n0 + wn * 32 + j * 8 + 2 * (lane & 3);
            if (r >= M || c >= N) continue;
            float x = acc[j][2 * h], y = acc[j][2 * h + 1];
            const size_t at = (size_t)r * N + c;
            if (ep.bias) {
                x += ep.bias[c];
                y += ep.bias[c + 1];
            }
            if (ep.relu) {
                x = fmaxf(x, 0.f);
                y = fmaxf(y, 0.f);
            }
            if (ep.mask) {
                const float2 k = *reinterpret_cast<const float2*>(ep.mask + at);
                x = k.x > 0.f ? x : 0.f;
                y = k.y > 0.f ? y : 0.f;
            }
            if (C) *reinterpret_cast<float2*>(C + at) = make_float2(x, y);
            if (ep.copy) *reinterpret_cast<__nv_bfloat162*>(ep.copy + at) = __floats2bfloat162_rn(x, y);
            if (ep.outer) {
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const float f = ep.m6[6 * r + k];
                    *reinterpret_cast<__nv_bfloat162*>(ep.outer + (size_t)(6 * r + k) * N + c) =
                        __floats2bfloat162_rn(f * x, f * y);
                }
            }
        }
}

// The elementwise step of a layer on its stored product, four columns per thread (N a multiple of 8)
__global__ void mlp_epilogue_kernel(float* C, size_t n4, int N, const MlpEpilogue ep)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 x = reinterpret_cast<const float4*>(C)[i];
        if (ep.bias) {
            const float* b = ep.bias + 4 * i % N;
            x = make_float4(x.x + b[0], x.y + b[1], x.z + b[2], x.w + b[3]);
        }
        if (ep.relu) x = make_float4(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f), fmaxf(x.z, 0.f), fmaxf(x.w, 0.f));
        if (ep.mask) {
            const float4 k = reinterpret_cast<const float4*>(ep.mask)[i];
            x = make_float4(k.x > 0.f ? x.x : 0.f, k.y > 0.f ? x.y : 0.f, k.z > 0.f ? x.z : 0.f, k.w > 0.f ? x.w : 0.f);
        }
        reinterpret_cast<float4*>(C)[i] = x;
        if (ep.copy) {
            reinterpret_cast<__nv_bfloat162*>(ep.copy)[2 * i] = __floats2bfloat162_rn(x.x, x.y);
            reinterpret_cast<__nv_bfloat162*>(ep.copy)[2 * i + 1] = __floats2bfloat162_rn(x.z, x.w);
        }
    }
}

// Whether a product runs in 32 x 64 tiles, by how many CTAs that takes.  The device holds three per SM at
// once; past that the general kernels' larger tiles pay, the deeper the product the sooner.  General kernel
// and element-wise step / this one (one GB300, 152 SMs; CTAs x K): rows [M][K] times [K][N] 768 x 4096 1.04,
// 768 x 512 1.25, 1024 x 512 0.92 .. 1.03, 1024 x 4096 0.80, 32768 x 256 1.16, 32768 x 4096 0.61; weight
// gradients (A transposed) 576 x 4096 1.02, 768 x 1024 0.95, 1024 x 1024 0.72; B transposed (tcgen05) 384 x
// 4096 1.00, 576 x 768 1.00, 768 x 512 1.23, 1024 x 512 0.95, 1536 x 256 1.00, 4096 x 64 1.10, 2048 x 4096 0.30.
// The outer product's six copies are worth the epilogue at every size (32768 x 4096: 0.95).
cudaError_t small_layer(int M, int N, int K, bool a_t, bool b_nk, const MlpEpilogue& ep, bool* small)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long ctas = (long long)((M + LM - 1) / LM) * ((N + LN - 1) / LN);
    if (ep.outer) *small = true;
    else if (a_t) *small = ctas <= 4LL * sms;
    else if (b_nk) *small = ctas <= 3LL * sms || ctas * K <= 2560LL * sms;
    else *small = ctas <= 6LL * sms || K <= 256;
    return e;
}

template <bool AT, bool BNK>
cudaError_t launch_layer(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, float* C,
                         const MlpEpilogue& ep, cudaStream_t st)
{
    constexpr int bytes = LayerTile<AT, BNK>::BYTES;
    const cudaError_t e = cudaFuncSetAttribute(layer_kernel<AT, BNK>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    const long long ctas = (long long)((M + LM - 1) / LM) * ((N + LN - 1) / LN);
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    layer_kernel<AT, BNK><<<(unsigned)ctas, LTHREADS, bytes, st>>>(M, N, K, A, lda, B, ldb, C, ep);
    return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_layer(int M, int N, int K, const __nv_bfloat16* A, int lda, bool a_t, const __nv_bfloat16* B, int ldb,
                       bool b_nk, float* C, const MlpEpilogue& ep, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (N % 8 || (a_t && b_nk) || (!C && !ep.outer)) return cudaErrorInvalidValue;
    bool small = true;
    cudaError_t e = small_layer(M, N, K, a_t, b_nk, ep, &small);
    if (e != cudaSuccess) return e;
    if (!small) {
        e = gemm_bf16(M, N, K, A, lda, a_t, B, ldb, b_nk, C, N, 1.f, 0.f, 1, st);
        if (e != cudaSuccess || !(ep.bias || ep.relu || ep.mask || ep.copy)) return e;
        const size_t n4 = (size_t)M * N / 4;
        const size_t blocks = (n4 + 255) / 256;
        mlp_epilogue_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(C, n4, N, ep);
        return cudaGetLastError();
    }
    if (a_t) return launch_layer<true, false>(M, N, K, A, lda, B, ldb, C, ep, st);
    if (b_nk) return launch_layer<false, true>(M, N, K, A, lda, B, ldb, C, ep, st);
    return launch_layer<false, false>(M, N, K, A, lda, B, ldb, C, ep, st);
}

cudaError_t gemm_bf16(int M, int N, int K, const __nv_bfloat16* A, int lda, bool a_t, const __nv_bfloat16* B,
                      int ldb, bool b_nk, float* C, int ldc, float alpha, float beta, int split_k, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (!a_t && b_nk) return gemm_bf16_tc(M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, split_k, st);
    if (split_k < 1) split_k = 1;
    int kps = (K + split_k - 1) / split_k;
    kps = (kps + BK - 1) / BK * BK;
    split_k = (K + kps - 1) / kps;
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, split_k);
    if (split_k > 1 && beta != 1.f) {
        // atomics add onto C: scale it first
        cudaError_t e = scale_f32(C, M, N, ldc, beta, st);
        if (e != cudaSuccess) return e;
    }
    if (!a_t && !b_nk) gemm_bf16_kernel<false, false><<<grid, THREADS, 0, st>>>(M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, kps);
    else if (a_t && b_nk) gemm_bf16_kernel<true, true><<<grid, THREADS, 0, st>>>(M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, kps);
    else gemm_bf16_kernel<true, false><<<grid, THREADS, 0, st>>>(M, N, K, A, lda, B, ldb, C, ldc, alpha, beta, kps);
    return cudaGetLastError();
}

}  // namespace es
