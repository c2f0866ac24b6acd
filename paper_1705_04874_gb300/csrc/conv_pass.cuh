// Derivative passes for axis lengths without an FFT plan (100, 190, the paper's
// 301 = 7 x 43, ...) as zero-padded convolutions.  Along a periodic axis the
// operator is a real circulant matrix, (D f)_i = sum_j c[(i - j) mod n] f_j, and
// the lags i - j run from -(n-1) to n-1: with the pencil padded by zeros to m >=
// 2 n - 1 points, the cyclic convolution of length m with the kernel laid out
// over those lags gives exactly these n sums, whatever the factors of n.  So the
// pass is the FFT pass of fft_pass.cuh with transforms of a length m that has a
// plan, a multiplier that is the m-point transform of the (far) kernel, n rows
// of input and n of output; the kernel is real, so two pencils still share a
// complex line.  The near stencil is longer (CONV_TAPS, es_internal.h) and wraps at n.
//
// Against the direct O(n) sum (circ_pass.cu, which the shortest axes and the
// compensated mode keep) the work per cell falls from n multiply-adds to about
// 5 log2 m operations, twice.  190^3 (m = 400), velocity / stress pass: x 0.312 /
// 0.335 -> 0.211 / 0.221 ms, y and z 0.288 / 0.303 -> 0.166 / 0.176 ms; the
// 301-cell z axis of the 125 x 75 x 301 grid (m = 625): 0.176 / 0.187 -> 0.086 /
// 0.092 ms.  What bounds them is the shared memory a tile takes ((m + 2 n) rows) and
// the registers of the radix-16 to 25 stages, which leave the y and z passes 4 CTAs on
// an SM (160 points), 3 (256, 320 and 400), 2 (500 and 625) or one (1024 points, every
// axis from 313 cells on: 130 to 156 KB), and the padded half of the transforms.  Even
// the one is ahead of the direct sum, ps per cell, velocity / stress: y and z 313 cells
// 55 / 58 -> 39 / 41, 400 64 / 69 -> 32 / 34, 512 72 / 74 -> 26 / 28; x 313 64 / 67 ->
// 44 / 46, 512 125 / 133 -> 34 / 36.
//
// A CTA keeps the arriving tile (n rows), the FFT's rows (m) and the near parts
// (n) in shared memory and is persistent, as the y and z passes are; the next
// tile starts to arrive when the first forward stage has read the current one.
#pragma once
#include "conv_plans.h"
#include "fft_pass.cuh"

namespace es {

template <> struct Dft<20> : DftPQ<4, 5> {};

template <int T, int PR>
__host__ __device__ constexpr int conv_threads() { return T * PR; }
// positions per thread outside the FFT, which deal the len / 2 cells an axis may have over the
// threads (in whole batches of the epilogue)
template <int M, int T>
__host__ __device__ constexpr int conv_rows()
{
    constexpr int r = (M / 2 + T - 1) / T;
    return r == 13 ? 15 : r;
}
template <int RA, int RB, int RC, int T, int PR>
__host__ __device__ constexpr int conv_min_blocks()
{
    constexpr int top = RA > RB ? RA : RB;
    constexpr int per_sm = top > 20 ? 448 : (top > 16 ? 512 : (top > 10 ? 768 : 1024));
    constexpr int b = per_sm / ((conv_threads<T, PR>() + 31) / 32 * 32);
    return b < 1 ? 1 : (b > 16 ? 16 : b);
}
template <int M, int PR>
__host__ __device__ constexpr size_t conv_smem(int n)
{
    return sizeof(float2) * ((size_t)M * PR + 2 * (size_t)n * PR + 3 * (size_t)M);
}
// x pass: the FFT's rows (at least n of them, from which the tile goes out in memory order) and
// the near parts
template <int M, int PR>
__host__ __device__ constexpr size_t conv_smem_x(int n)
{
    return sizeof(float2) * ((size_t)M * PR + (size_t)n * PR + 2 * (size_t)M);
}

// near_part for an axis length known at run time, R rows from e0 on, wrapped at n: every row that is
// read goes to all the sums that it has a tap in, so that R sums are live and not CONV_TAPS rows
template <int R, class Row, class Put>
__device__ __forceinline__ void near_part_n(const PassJob& J, int e0, int n, Row row, Put put)
{
    const int ofs = conv_near_ofs(J.sign);
    float2 s[R];
#pragma unroll
    for (int q = 0; q < R; ++q) s[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < R + CONV_TAPS - 1; ++k) {
        int e = e0 + ofs + k;
        e = e < 0 ? e + n : e;
        e = e >= n ? e - n : e;
        const float2 w = e < n ? row(e) : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (k >= q && k - q < CONV_TAPS) s[q] = fma2(rep2(J.g[k - q]), w, s[q]);
        if (k >= CONV_TAPS - 1 && e0 + k - (CONV_TAPS - 1) < n) put(e0 + k - (CONV_TAPS - 1), s[k - (CONV_TAPS - 1)]);
    }
}

// y and z passes (see pass_strided): n = p.n cells through an FFT of M points
template <int RA, int RB, int RC, int T, int PR, int V>
__global__ void __launch_bounds__(conv_threads<T, PR>(), conv_min_blocks<RA, RB, RC, T, PR>())
conv_strided(const __grid_constant__ PassParams p, int ntiles)
{
    using C = CoreOf<RA, RB, RC, T, PR>;
    constexpr int M = C::N, NT = T * PR, RN = conv_rows<M, T>();
    extern __shared__ __align__(16) float2 smem[];
    const int n = p.n;
    float2* tile = smem;           // the arriving tile
    float2* buf = tile + n * PR;   // the FFT's rows
    float2* nearp = buf + M * PR;  // near parts
    float2* s_tw = nearp + n * PR;
    float2* s_hp = s_tw + M;
    float2* s_hm = s_hp + M;
    const int tid = threadIdx.x;
    const int c = tid % PR, j = tid / PR;
    pdl_begin(p.pdl);
    const unsigned est = p.axis == 1 ? (unsigned)p.nx : (unsigned)p.nx * p.ny;
    const int total = ntiles * p.njobs;
    auto stage = [&](const StridedTile& t) {
        if (V == 1) stage_strided<NT, 1, PR>(p, t, tile, est, n);
        else if (p.nx % 4 == 0) stage_strided<NT, 4, PR>(p, t, tile, est, n);
        else stage_strided<NT, 2, PR>(p, t, tile, est, n);
    };
    stage(strided_tile<PR>(p, blockIdx.x, ntiles));
    for (int i = tid; i < M; i += NT) {
        s_tw[i] = __ldg(p.tw + i);
        s_hp[i] = __ldg(p.hp + i);
        s_hm[i] = __ldg(p.hm + i);
    }
    bool waited = p.pdl != 1;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        const PassJob& J = p.job[w / ntiles];
        cp_async_commit_wait_all();
        __syncthreads();  // the tile is there; the previous one's rows are no longer read
        if (J.coef[0]) {  // coefficient and PML slab rows into L2 for the epilogue
            const StridedTile t = strided_tile<PR>(p, w, ntiles);
            for (int i = tid; i < n; i += NT) {
                const unsigned o = (unsigned)i * est;
                if (ES_INB(p, t.base + o, p.ext_c)) {
                    prefetch_l2(J.coef[0] + t.base + o);
                    if (J.coef[1]) prefetch_l2(J.coef[1] + t.base + o);
                }
            }
            const size_t s0 = t.soff + t.x0 + (p.axis == 1 ? (size_t)p.nx * p.S * t.outer : (size_t)p.nx * t.outer);
            for (int i = tid; i < p.S; i += NT) {
                const unsigned o = (unsigned)i * est;
                if (ES_INB(p, s0 + o, p.ext_s)) {
                    prefetch_l2(J.slab[0] + s0 + o);
                    if (J.coef[1]) {
                        prefetch_l2(J.slab[1] + s0 + o);
                        prefetch_l2(J.slab[2] + s0 + o);
                    }
                }
            }
        }
        if (RN * j < n)
            near_part_n<RN>(
                J, RN * j, n, [&](int e) { return tile[e * PR + c]; },
                [&](int e, float2 s) { nearp[e * PR + c] = s; });
        {
            float2 a[C::MA][RA];
            C::stageA(a, j, [&](int e) { return e < n ? tile[e * PR + c] : make_float2(0.f, 0.f); });
            C::stageA_store(a, buf, j, c);
            __syncthreads();  // the rows are there; the tile has been read
            if (w + (int)gridDim.x < total) stage(strided_tile<PR>(p, w + gridDim.x, ntiles));
            C::middle(buf, s_tw, J.sign > 0 ? s_hp : s_hm, j, c);
            __syncthreads();
            C::stageA_inv(buf, s_tw, a, j, c);
            __syncthreads();  // the FFT's rows have been read
            C::results(a, j, [&](int e, float2 v) {
                if (e < n) buf[e * PR + c] = v;
            });
        }
        const StridedTile t = strided_tile<PR>(p, w, ntiles);
        StridedEpilogue<RN, V, false, false, PR> ep(p, J, t, est, buf, nearp, 0);
        ep.first_coefs();
        __syncthreads();  // the far parts are there
        if (!waited) {
            pdl_wait();  // the previous pass's updates of the targets come first
            waited = true;
        }
        if (J.kind == JOB_STORE) ep.template run<JOB_STORE, false>();
        else if (J.kind == JOB_SINGLE) ep.template run<JOB_SINGLE, true>();
        else ep.template run<JOB_NORMAL, true>();
        if (p.L > 0 && J.kind != JOB_STORE) {
            __syncthreads();
            if (J.kind == JOB_SINGLE) ep.template run_slab<JOB_SINGLE, NT>();
            else ep.template run_slab<JOB_NORMAL, NT>();
        }
    }
}

// x pass: a tile is 2 PR consecutive x-lines, one contiguous block of memory;
// blockIdx.y = job.  Staged and turned around four lines x eight cells per warp
// (any length, any alignment); the derivatives go back to memory order through
// the FFT's rows and out four cells per thread (x_quads).
template <int PR>
__device__ __forceinline__ int conv_x_swz(int x)
{
    return PR == 16 ? (x & 7) << 1 : ((x >> 1) & 3) << 1;
}
template <int RA, int RB, int RC, int T, int PR>
__global__ void __launch_bounds__(conv_threads<T, PR>(), conv_min_blocks<RA, RB, RC, T, PR>())
conv_x(const __grid_constant__ PassParams p)
{
    using C = CoreOf<RA, RB, RC, T, PR>;
    constexpr int M = C::N, NT = T * PR, RN = conv_rows<M, T>(), LINES = 2 * PR, LG = LINES / 4;
    extern __shared__ __align__(16) float2 smem[];
    const int n = p.n;
    float2* buf = smem;
    float2* nearp = buf + M * PR;
    float2* s_tw = nearp + n * PR;
    float2* s_h = s_tw + M;
    float* bf = reinterpret_cast<float*>(buf);
    const int tid = threadIdx.x;
    const int c = tid % PR, j = tid / PR;
    const PassJob& J = p.job[blockIdx.y];
    pdl_begin(p.pdl);
    const int nlines = p.ny * p.nz;
    const int sim = blockIdx.x % p.nsim;
    const size_t off = (size_t)sim * p.fstride, soff = (size_t)sim * p.sstride;
    const int line0 = (int)(blockIdx.x / p.nsim) * LINES, nl = min(LINES, nlines - line0);
    const size_t q0 = (size_t)line0 * n;
    const float* src = J.src + off + q0;
    // warp item: lines 4 lg .. 4 lg + 3, cells 8 xb .. 8 xb + 7
#pragma unroll 2
    for (int it = tid; it < LG * 32 * ((n + 7) / 8); it += NT) {
        const int wi = it / 32, r = 4 * (wi % LG) + (it / 8) % 4, xx = 8 * (wi / LG) + it % 8;
        if (xx >= n) continue;
        const bool ok = r < nl && ES_INB(p, off + q0 + r * n + xx, p.ext_f);
        cp_async<4>(bf + xx * LINES + (r ^ (conv_x_swz<PR>(xx) << 1)), ok ? src + r * n + xx : src, ok);
    }
    if (J.coef[0])  // the tile's coefficient lines (contiguous) into L2
        for (int f = 32 * tid; f < nl * n; f += 32 * NT) {
            prefetch_l2(J.coef[0] + q0 + f);
            if (J.coef[1]) prefetch_l2(J.coef[1] + q0 + f);
        }
    const float2* h = J.sign > 0 ? p.hp : p.hm;
    for (int i = tid; i < M; i += NT) {
        s_tw[i] = __ldg(p.tw + i);
        s_h[i] = __ldg(h + i);
    }
    cp_async_commit_wait_all();
    __syncthreads();
    auto at = [&](int e) { return e * PR + (c ^ conv_x_swz<PR>(e)); };
    if (RN * j < n)
        near_part_n<RN>(
            J, RN * j, n, [&](int e) { return buf[at(e)]; }, [&](int e, float2 s) { nearp[e * PR + c] = s; });
    float2 a[C::MA][RA];
    C::stageA(a, j, [&](int e) { return e < n ? buf[at(e)] : make_float2(0.f, 0.f); });
    __syncthreads();  // the staged rows have been read; the near parts are visible
    C::stageA_store(a, buf, j, c);
    __syncthreads();
    C::middle(buf, s_tw, s_h, j, c);
    __syncthreads();
    C::stageA_inv(buf, s_tw, a, j, c);
    __syncthreads();  // the FFT's rows have been read
    C::results(a, j, [&](int e, float2 v) {
        if (e >= n) return;
        const float2 s = nearp[e * PR + c];
        float* o = bf + 2 * c * n + e;  // lines 2c, 2c + 1 in memory order
        o[0] = __fadd_rn(v.x, s.x);
        o[n] = __fsub_rn(s.y, v.y);
    });
    __syncthreads();
    if (p.pdl == 1) pdl_wait();  // the previous pass's updates of the targets come first
    const int nf = nl * n;
    const XQuads xq = x_quads(J, off, q0, nf);
    const float inv = 1.f / (float)n;
    // line of the tile's cell f: floor((f + 1/2) / n), exact for these f < 2^15 (the nearest
    // multiple of 1 / n is at least 1 / (2 n) away, far above the rounding)
    auto line_of = [&](int f) { return (int)(((float)f + 0.5f) * inv); };
    x_quads_update<NT>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    // what is left: the cells before the first chunk and past the last one
    for (int i = tid; i < nf - 4 * xq.nq; i += NT) {
        const int f = i < xq.h ? i : i + 4 * xq.nq, r = line_of(f), x = f - r * n, line = line0 + r;
        // the slab index along x is sp + S (y + ny z) = sp + S line: the line goes in as y, with z = 0
        epilogue_one(p, J, q0 + f, x, x, line, 0, bf[f], off, soff);
    }
}

template <int RA, int RB, int RC, int T, int PR, int V>
static cudaError_t launch_conv_strided(const PassParams& p, cudaStream_t st)
{
    constexpr int threads = conv_threads<T, PR>(), W = 2 * PR;
    const size_t smem = conv_smem<RA * RB * RC, PR>(p.n);
    const int ntiles = (p.nx + W - 1) / W * (p.axis == 1 ? p.nz : p.ny) * p.nsim;
    int grid = 0;
    const cudaError_t e = persistent_grid(conv_strided<RA, RB, RC, T, PR, V>, threads, smem, ntiles * p.njobs, &grid);
    if (e != cudaSuccess) return e;
    return launch_pass_kernel(conv_strided<RA, RB, RC, T, PR, V>, dim3((unsigned)grid), threads, smem, st, p, ntiles);
}

template <int RA, int RB, int RC, int T, int PR, int V>
static cudaError_t prepare_conv_strided()
{
    return cudaFuncSetAttribute(conv_strided<RA, RB, RC, T, PR, V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)conv_smem<RA * RB * RC, PR>(RA * RB * RC / 2));
}

}  // namespace es
