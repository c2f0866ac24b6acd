// Internal declarations of the surrogate network's kernels (not public ABI).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace es {

// C[M][N] = alpha op(A) op(B) + beta C (BF16 operands, FP32 accumulate); see
// sur_gemm.cu.  Leading dimensions and K multiples of 8.
cudaError_t gemm_bf16(int M, int N, int K, const __nv_bfloat16* A, int lda, bool a_t, const __nv_bfloat16* B,
                      int ldb, bool b_nk, float* C, int ldc, float alpha, float beta, int split_k, cudaStream_t st);

// What a layer of the encoder does with its product x (row r, column c), in this order; null: not
struct MlpEpilogue {
    const float* bias = nullptr;      // x += bias[c]
    bool relu = false;                // x = max(x, 0)
    const float* mask = nullptr;      // x = 0 where mask[r][c] <= 0
    __nv_bfloat16* copy = nullptr;    // BF16 copy [M][N]
    const float* m6 = nullptr;        // with outer: outer[r][k N + c] = m6[r][k] x, k < 6 (BF16)
    __nv_bfloat16* outer = nullptr;
};
// C[M][N] = op(A) op(B) through the epilogue (N a multiple of 8; C may be null with an outer product), for
// products too small to fill the device in 128 x 128 tiles by layer_kernel in sur_gemm.cu, the others by the
// general kernels
cudaError_t gemm_layer(int M, int N, int K, const __nv_bfloat16* A, int lda, bool a_t, const __nv_bfloat16* B, int ldb,
                       bool b_nk, float* C, const MlpEpilogue& ep, cudaStream_t st);

// the K-major case (A [M][K], B [N][K]) on tcgen05 tensor cores; see sur_gemm_tc.cu.
// alpha4 (host, 4 values) with span > 0: column n of C takes alpha4[n / span] instead of
// alpha (4 span >= N), e.g. one scale per output component of the decoder
cudaError_t gemm_bf16_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb,
                         float* C, int ldc, float alpha, float beta, int split_k, cudaStream_t st,
                         const float* alpha4 = nullptr, int span = 0);
// The Adam step of a row-major weight block W[M][N] (p, its moments m, v) with the gradient A[M][K]
// B[N][K]^T taken from tensor memory and never stored; writes the BF16 copy row-major (pb) and
// transposed (pt, [N][M]).  N a multiple of 8, arrays 16-byte aligned; see sur_gemm_tc.cu.
cudaError_t gemm_adam_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, float* p,
                         float* m, float* v, float lr, float b1, float b2, float eps, int t, __nv_bfloat16* pb,
                         __nv_bfloat16* pt, cudaStream_t st);
// reads and clears the tcgen05 GEMM's device status word (bits set by waits that gave up)
cudaError_t gemm_tc_status(unsigned* status);
// Launches one kernel whose bounded wait on a barrier nothing completes gives
// up after `seconds` (0 < seconds <= 2) and sets the status word.
cudaError_t gemm_wait_probe(double seconds, cudaStream_t st);
// The give-up path of a pair of CTAs: one pair on a 256 x 256 x 1280 product of zeros whose producer in
// CTA `rank` stops before k-block `stage` < 20, the other waits running out after 50 ms; synchronizes
// and returns the status word (not cleared): bits 3 and 4 stay clear if the copies were all awaited.
cudaError_t gemm_pair_probe(int rank, int stage, unsigned* status, cudaStream_t st);
// out[c][r] = in[r][c] for a rows x cols BF16 matrix (row-major both)
cudaError_t transpose_bf16(const __nv_bfloat16* in, long long rows, long long cols, __nv_bfloat16* out,
                           cudaStream_t st);

cudaError_t scale_f32(float* C, int M, int N, int ldc, float s, cudaStream_t st);
cudaError_t cast_bf16(const float* x, __nv_bfloat16* y, size_t n, cudaStream_t st);
// position features: [p, sin(2^j pi p), cos(2^j pi p)], j < nfreq, zero padded to width
cudaError_t sur_features(const float* pos, int B, int nfreq, int width, __nv_bfloat16* X, cudaStream_t st);
// dA[b][k] = sum_c M[b][c] dZ[b][c K + k], FP32 and BF16
cudaError_t sur_contract(const float* M6, const float* dZ, int B, int K, float* dA, __nv_bfloat16* dAb,
                         cudaStream_t st);
// outputs [B][4][Dc], y = scale[c] u, tau = t / scale[c]: per sample
// l_b = sum_c |u_c - tau_c|^2 / (sum_c |tau_c|^2 + eps) (squared relative L2 of
// the component-scaled seismogram), loss = mean_b l_b (device float),
// per_sample (optional, device [B]) = l_b, dU = dloss/du in BF16 and dUT its
// transpose (skipped when null); Dc and B multiples of 8; acc: device scratch of 8 B floats, 8-byte aligned
cudaError_t sur_loss(const float* U, const float* T, const float* scale, int B, long long Dc, float eps,
                     __nv_bfloat16* dU, __nv_bfloat16* dUT, float* loss, float* acc, float* per_sample, cudaStream_t st);
cudaError_t sur_init_normal(float* p, size_t n, float std, unsigned long long seed, cudaStream_t st);
// ss[c] = sum of squares of component c over n samples [n][4][Dc]
cudaError_t sur_comp_sumsq(const float* T, int n, long long Dc, float* ss, cudaStream_t st);
// out[b] = sum_c mt[b][c] G[loc[b]][c] (G: [n_loc][6][D])
cudaError_t sur_combine(const float* G, long long D, const int* loc, const float* mt, int B, float* out,
                        cudaStream_t st);
// db[n] = sum_b G[b][n]
cudaError_t sur_colsum(const float* G, int B, int N, float* db, cudaStream_t st);
// Adam step (bias-corrected, lr, b1, b2, eps) on FP32 params, refreshing the BF16 copy (may be null)
cudaError_t sur_adam(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2, float eps,
                     int t, __nv_bfloat16* pb, cudaStream_t st);

// The same step on a row-major [rows][cols] block (the decoder; both multiples of 4, 16-byte aligned),
// writing the BF16 copy both row-major (pb) and transposed (pt, [cols][rows])
cudaError_t sur_adam_t(float* p, const float* g, float* m, float* v, long long rows, long long cols, float lr, float b1,
                       float b2, float eps, int t, __nv_bfloat16* pb, __nv_bfloat16* pt, cudaStream_t st);

}  // namespace es
