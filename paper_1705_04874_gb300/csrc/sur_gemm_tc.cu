// BF16-input, FP32-accumulate GEMM on the fifth-generation tensor cores
// (tcgen05) for the K-major storage order of both operands:
//   C[M][N] = alpha * A[M][K] * B[N][K]^T + beta * C
// A row-major [M][K] (lda), B row-major [N][K] (ldb), C FP32 row-major (ldc).
//
// Persistent: one CTA per SM (or pairs of them, below) walks the 128 x 256 output
// tiles (x split_k slices of K) with stride gridDim.x, 6 warps:
//   warp 0, one thread: TMA producer -- 64-wide K slabs of A (128 rows) and
//       B (256 rows) into a 4-stage ring of 128-byte-swizzled shared tiles,
//       completion tracked by transaction-count mbarriers; it runs ahead
//       across tile boundaries;
//   warp 1, one thread: issues tcgen05.mma (M 128, N 256, K 16; both
//       operands from shared-memory descriptors) into one of two 256-column
//       FP32 accumulators in tensor memory (512 columns); tcgen05.commit
//       frees each stage and, at the end of a tile, hands the accumulator to
//       the epilogue;
//   warps 2-5: epilogue -- warp w owns TMEM lanes (tile rows)
//       32 (w mod 4) .. +31, reads 32 columns at a time with tcgen05.ld
//       (lane = row), turns the 32 x 32 block around in its own shared
//       buffer so that each store instruction covers four whole 128-byte row
//       segments, and writes alpha * acc + beta * C (split_k > 1: atomically
//       adds alpha * acc onto a C that already holds beta * C), then returns
//       the accumulator; the next tile's MMAs run in the other one meanwhile.
// With an even number of row tiles, and enough work (PAIR_MIN_K, PAIR_MIN_WORK), two
// CTAs (a cluster) work on two of them as one
// 256 x 256 tile: each loads its 128 rows of A and half of B's rows, the first one's
// issuer runs tcgen05.mma.cta_group::2 (M 256) over both, and each reads its own
// 128 rows back.  Shared memory is what bounds a CTA on its own: it must take in
// and give to the tensor core 384 rows per 64 of K, a CTA of a pair 256 (and the
// ring is 6 stages deep in the same memory).  One GB300, N = 262144, K = 4608:
// 256 rows 504 -> 443 us; 1024 rows, a serving batch with its encoder 1.78 -> 1.69
// ms; 256 x 4608 with K = 262144 in 128 slices 560 -> 477 us.  (The pair sharing B by
// TMA multicast alone, each CTA with its own MMAs: 506, 1.80 and 544.)  An odd
// number of row tiles stays with single CTAs: a pair's empty half is work for
// nothing, half of it all at a single row tile.
// Rows, columns and K past the matrix edge are zero-filled by TMA and masked
// in the epilogue.  Every mbarrier wait gives up after WAIT_NS of global
// time, records the role that gave up in a device status word (read and
// cleared by gemm_tc_status) and lets the CTA finish: the MMAs issued are
// awaited, TMA copies still in flight are awaited (both bounded) and the
// tensor memory is always freed.  A pair's copies are counted stage by stage by
// the first CTA's barriers, which complete when both CTAs' shares have landed: at
// the end the CTAs compare how many stages each has started, the one that gave up
// earlier starts the missing ones too (nothing reads them any more), and the first
// one waits for them all before either leaves.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "sur_adam.cuh"
#include "sur_internal.h"
#include "tc_ptx.cuh"

namespace es {
namespace {

using namespace tcx;

constexpr int TM = 128;  // tile rows = MMA M = TMEM lanes
constexpr int TN = 256;  // tile columns = MMA N = TMEM columns (FP32)
constexpr int TK = 64;   // K per stage: one 128-byte swizzle row of BF16
constexpr int UK = 16;   // K of one tcgen05.mma kind::f16
constexpr int STAGES = 4;
constexpr int A_BYTES = TM * TK * 2;
constexpr int B_BYTES = TN * TK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int EPI_LD = 36;  // row stride (floats) of an epilogue warp's 32 x 32 staging block: 16-byte rows
constexpr int EPI_BYTES = 4 * 32 * EPI_LD * 4;
// ring + staging + alignment slack for the 1024-byte swizzle atoms
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 1024;
constexpr int THREADS = 192;
constexpr unsigned TMEM_COLS = 2 * TN;  // two accumulators

static_assert(A_BYTES % 1024 == 0 && STAGE_BYTES % 1024 == 0, "swizzle atoms must stay 1024-byte aligned");
static_assert(TK == 64, "make_map boxes are 64 BF16 wide");

// instruction descriptor for kind::f16: D FP32 (bits 4-5 = 1), A BF16 (bits
// 7-9 = 1), B BF16 (bits 10-12 = 1), both K-major (bits 15, 16 = 0), N / 8 in
// bits 17-22, M / 16 in bits 24-28
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) |
                           ((uint32_t)(TM >> 4) << 24);

// of a pair of CTAs: M is that of both
constexpr uint32_t IDESC_PAIR = (IDESC & ~(0x1fu << 24)) | ((uint32_t)(2 * TM >> 4) << 24);
// Pairs where a tile has PAIR_MIN_K k-blocks or more and each SM's share of all tiles' k-blocks is at
// least PAIR_MIN_WORK.  A pair costs 1 to 2 us a launch (the cluster's launch and its two barriers), and
// with few k-blocks a tile is bound by its output, not its operands.  us, single CTAs and pairs (one GB300;
// tiles x k-blocks): 2 x 4 10.8 and 12.5, 512 x 12 37.1 and 37.3, 2048 x 12 104 and 103, 384 x 16 30.6 and
// 30.9, 608 x 16 41.7 and 39.7, 1024 x 16 65.8 and 61.2, 256 x 24 28.9 and 28.7, 512 x 24 55.4 and 48.4, 64 x
// 72 31.0 and 33.0, 152 x 72 41.0 and 37.1, 512 x 72 125 and 105; past both lines pairs won every one of 108
// sizes but one (16 x 128 k-blocks in 8 row tiles, 2 % lost), by 14 % on average.
constexpr int PAIR_MIN_K = 16, PAIR_MIN_WORK = 64;
// a CTA of a pair holds half of B's rows, so the ring is deeper
template <int CL>
__host__ __device__ constexpr int tc_stages() { return STAGES * STAGE_BYTES / (A_BYTES + B_BYTES / CL); }

__device__ unsigned g_tc_status;  // bit 0 producer, 1 MMA, 2 epilogue, 3 MMA drain, 4 TMA drain, 5 probe gave up

// The timeout path of the bounded waits, on demand: one thread waits, through
// mbar_wait, on the first phase of a fresh barrier that nothing arrives at,
// gives up after limit_ns, records bit 5 of the status word and returns.
__global__ void wait_probe_kernel(unsigned long long limit_ns)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!mbar_wait(&bar, 0, limit_ns)) atomicOr(&g_tc_status, 32u);
    }
}

// PROBE (pairs): the producer of CTA `span` mod 2 gives up before its stage `span` / 2, as after a wait
// that ran out, and the other roles' waits run out after PROBE_NS (gemm_pair_probe)
constexpr unsigned long long PROBE_NS = 50000000ull;
template <int CL, bool PROBE = false>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int M, int N,
                   int nkb, int kb_per, int mt, int ntl, int ntiles, float* __restrict__ C, int ldc, float alpha,
                   float beta, int atomic, float4 alpha4, int span)
{
    constexpr unsigned long long LIMIT = PROBE ? PROBE_NS : WAIT_NS;
    extern __shared__ uint8_t dyn[];
    constexpr int ST = tc_stages<CL>(), BYTES = A_BYTES + B_BYTES / CL;  // a stage of this CTA
    __shared__ __align__(8) uint64_t full[ST], empty[ST], acc_full[2], acc_empty[2], mma_done;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_issued, s_consumed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(dyn) + 1023u) & ~1023u;
    // CTA r of a cluster takes row tile CL p + r of the cluster's tiles
    const int r = CL > 1 ? (int)cluster_rank() : 0;
    ntiles /= CL;
    mt /= CL;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4 * CL);  // one arrival per epilogue warp of the cluster
        }
        mbar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    __syncwarp();
    if (warp == 0) {
        if constexpr (CL == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (CL > 1) cluster_sync();  // the barriers of every CTA are there
    const uint32_t tmem = tmem_slot;
    auto commit = [](uint64_t* bar) {
        if constexpr (CL == 1) tc_commit(bar);
        else tc_commit_pair(bar);
    };
    // this CTA's copies into stage s: 64 of K from x on, A's rows from ya and B's from yb on
    auto load = [&](int s, int x, int ya, int yb) {
        const uint32_t sa = base + s * BYTES;
        if constexpr (CL == 1) {
            mbar_expect_tx(&full[s], BYTES);
            tma_load_2d(sa, &mapA, &full[s], x, ya);
            tma_load_2d(sa + A_BYTES, &mapB, &full[s], x, yb);
        } else {  // each CTA its rows of A and of B; the issuing CTA's barrier hears of both
            if (r == 0) mbar_expect_tx(&full[s], CL * BYTES);
            const uint32_t bar = cluster_addr(&full[s], 0);
            tma_load_2d_pair(sa, &mapA, bar, x, ya);
            tma_load_2d_pair(sa + A_BYTES, &mapB, bar, x, yb);
        }
    };

    if (warp == 0) {
        if (lane == 0) {
            // producer: every k-block of every tile of this CTA, through the ring
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x / CL; t < ntiles && ok; t += gridDim.x / CL) {
                const int mi = t % mt * CL + r, rest = t / mt;
                const int ni = rest % ntl, kb0 = (rest / ntl) * kb_per;
                const int nk = min(nkb, kb0 + kb_per) - kb0;
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const int s = it % ST;
                    if ((PROBE && span == 2 * it + r) || !mbar_wait(&empty[s], ((it / ST) & 1) ^ 1, LIMIT)) {
                        atomicOr(&g_tc_status, 1u);
                        ok = false;
                        break;
                    }
                    load(s, (kb0 + kb) * TK, mi * TM, ni * TN + r * (TN / CL));
                }
            }
            s_issued = it;
        }
    } else if (warp == 1) {
        if (lane == 0 && r == 0) {
            // MMA issuer (of a cluster: its first CTA's): accumulator b = local tile index mod 2
            int it = 0, lt = 0;
            bool ok = true;
            for (int t = blockIdx.x / CL; t < ntiles && ok; t += gridDim.x / CL, ++lt) {
                const int rest = t / mt;
                const int kb0 = (rest / ntl) * kb_per;
                const int nk = min(nkb, kb0 + kb_per) - kb0;
                const int b = lt & 1;
                if (!mbar_wait(&acc_empty[b], ((lt >> 1) & 1) ^ 1, LIMIT)) {
                    atomicOr(&g_tc_status, 2u);
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * TN);
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const int s = it % ST;
                    if (!mbar_wait(&full[s], (it / ST) & 1, LIMIT)) {
                        atomicOr(&g_tc_status, 2u);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = base + s * BYTES;
                    const uint64_t da = sw128_desc(sa), db = sw128_desc(sa + A_BYTES);
#pragma unroll
                    for (int k = 0; k < TK / UK; ++k) {
                        const uint64_t step = (uint64_t)((k * UK * 2) >> 4);  // 32 bytes along the swizzled row
                        if constexpr (CL == 1) tc_mma(acc, da + step, db + step, IDESC, (kb | k) != 0);
                        else tc_mma_pair(acc, da + step, db + step, IDESC_PAIR, (kb | k) != 0);
                    }
                    commit(&empty[s]);
                }
                if (ok) commit(&acc_full[b]);
            }
            s_consumed = it;
            commit(&mma_done);  // arrives when every MMA issued above has completed
        }
    } else {
        // epilogue warps 2..5: TMEM lane quarter q = warp mod 4
        const int q = warp & 3;
        const bool vec = (ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
        int lt = 0;
        for (int t = blockIdx.x / CL; t < ntiles; t += gridDim.x / CL, ++lt) {
            const int mi = t % mt * CL + r, ni = (t / mt) % ntl;
            const int b = lt & 1;
            // one lane waits and the warp follows its result: tcgen05.ld below needs the whole warp
            int got = 0;
            if (lane == 0) got = mbar_wait(&acc_full[b], (lt >> 1) & 1, LIMIT) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) atomicOr(&g_tc_status, 4u);
                break;
            }
            tc_fence_after();
            const int n0 = ni * TN, row0 = mi * TM + q * 32;
            // this warp's staging block: row r (TMEM lane) at stage + r * EPI_LD
            float* stage = reinterpret_cast<float*>(dyn + (base - smem_u32(dyn)) + ST * BYTES) +
                           q * 32 * EPI_LD;
            for (int c0 = 0; c0 < TN; c0 += 32) {
                if (n0 + c0 >= N) break;  // uniform over the warp
                __syncwarp();               // the previous block's reads of the staging rows are done
                uint32_t acc[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * TN + c0), acc);
                float4* srow = reinterpret_cast<float4*>(stage + lane * EPI_LD);
                // per-column alpha: columns [c span, (c + 1) span) of C take component c of alpha4, one choice
                // for a block that lies within a component (64 sources x 262144 outputs with 192 inputs, one
                // GB300: a serving batch 78 us, 137 and 151 with a choice per column)
                auto comp = [&](int col) { return (col >= span) + (col >= 2 * span) + (col >= 3 * span); };
                const int first = n0 + c0, c4 = !PROBE && span ? comp(first) : -1;
                const float one = c4 < 0 ? alpha : c4 == 0 ? alpha4.x : c4 == 1 ? alpha4.y : c4 == 2 ? alpha4.z : alpha4.w;
                if (c4 >= 0 && comp(first + 31) != c4) {  // (a block on a component's edge)
                    float a[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int col = n0 + c0 + j;
                        a[j] = (col < span ? alpha4.x : col < 2 * span ? alpha4.y : col < 3 * span ? alpha4.z
                                                                                                  : alpha4.w) *
                               __uint_as_float(acc[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) srow[j] = make_float4(a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        srow[j] = make_float4(one * __uint_as_float(acc[4 * j]), one * __uint_as_float(acc[4 * j + 1]),
                                              one * __uint_as_float(acc[4 * j + 2]), one * __uint_as_float(acc[4 * j + 3]));
                }
                __syncwarp();
                // lane l stores columns 4 (l mod 8) .. +3 of row 4 i + l / 8: a warp instruction writes
                // four whole 128-byte row segments
                const int cc = n0 + c0 + 4 * (lane & 7);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = 4 * i + (lane >> 3), grow = row0 + rr;
                    if (grow >= M || cc >= N) continue;
                    float4 v = *reinterpret_cast<const float4*>(stage + rr * EPI_LD + 4 * (lane & 7));
                    float* p = C + (size_t)grow * ldc + cc;
                    if (vec && cc + 4 <= N) {
                        float4* dst = reinterpret_cast<float4*>(p);
                        if (atomic) {
                            atomicAdd(dst, v);
                        } else {
                            if (beta != 0.f) {
                                const float4 o = *dst;
                                v.x += beta * o.x;
                                v.y += beta * o.y;
                                v.z += beta * o.z;
                                v.w += beta * o.w;
                            }
                            *dst = v;
                        }
                    } else {
                        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (cc + k >= N) break;
                            if (atomic) atomicAdd(p + k, e[k]);
                            else p[k] = beta != 0.f ? e[k] + beta * p[k] : e[k];
                        }
                    }
                }
            }
            // every tcgen05.ld of this warp has completed (tmem_ld32 waits): hand the accumulator back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (CL == 1) mbar_arrive(&acc_empty[b]);
                else mbar_arrive_cluster(cluster_addr(&acc_empty[b], 0));
            }
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (CL > 1) cluster_sync();  // both producers have stopped
    if (threadIdx.x == 0) {
        if (!mbar_wait(&mma_done, 0)) atomicOr(&g_tc_status, 8u);
        // copies issued but never consumed (only after a wait gave up) must land before the CTA exits
        int issued = s_issued;
        if constexpr (CL > 1) {
            // stages the other CTA started alone: their places here are free (it saw them released by the
            // MMAs, which read both CTAs' memory)
            for (const int other = cluster_load(&s_issued, r ^ 1); issued < other; ++issued) load(issued % ST, 0, 0, 0);
        }
        for (int it = s_consumed; r == 0 && it < issued; ++it)
            if (!mbar_wait(&full[it % ST], (it / ST) & 1)) atomicOr(&g_tc_status, 16u);
    }
    __syncthreads();
    if (CL > 1) cluster_sync();  // no CTA leaves while another may write to it or to its barriers
    if (warp == 0) {
        tc_fence_after();
        if constexpr (CL == 1)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// ---------------------------------------------------------------------------
// dW = A B^T with the Adam step in the epilogue: the gradient of a weight block
// W[M][N] goes from tensor memory straight into the update of p, m and v, and of
// the two BF16 copies (row-major pb, transposed pt), and is never stored.
//
// What bounds it is HBM: 28 bytes per weight (p, m, v read and written, two BF16
// copies written) against 36 with the gradient written by one kernel and read by
// the next.  A tile is 128 x 128 and K is one batch: up to seven k-blocks (larger
// batches go to two kernels, adam_in_gemm in es_sur.cu) one operand stage is
// enough (the MMAs run a tile ahead of the epilogue) and the rest of shared
// memory moves the weights: each of eight epilogue warps walks
// 32 x 32 blocks of p, m and v through two places of its own, one block arriving
// by TMA while the other is updated in place and leaves by TMA.  A lane holds a
// row, as tcgen05.ld delivers the gradient, so nothing is turned around but the
// row-major BF16 copy: the 128-byte swizzle keeps the 16-byte accesses free of
// bank conflicts, and the transposed copy is written by columns (32 lanes, 64
// contiguous bytes).
// 4608 x 262144 weights, batch 256 (one GB300): 5.8 ms, 5.8 TB/s, where the two
// kernels took 7.0 (1.26 and 5.7, at 6.8 TB/s; 8.65 -> 7.46 ms per training
// step).  Of the step times on the way: operands through registers 10.5 (the
// kernel spilled, which waits for each load where it is issued), blocks of 16
// columns 9.0 (TMA moves a row of 64 bytes no faster than one of 128), the
// row-major copy stored 16 bytes a row 8.2, the two column blocks of a row not
// side by side 7.9; prefetching into L2 was slower (8.5).  Without the copies
// it runs at the same 5.8 TB/s: the rest is DRAM's rate for this pattern.
constexpr int AD_TN = 128, AD_STAGES = 1, AD_WARPS = 8, AD_THREADS = 32 * (2 + AD_WARPS);
constexpr int AD_STAGE_BYTES = A_BYTES + AD_TN * TK * 2;
constexpr int AD_COLS = 32, AD_RING = 2;             // columns of a block, blocks of a warp's ring
constexpr int AD_ARRAY = 32 * AD_COLS * 4;           // one array's block: 32 rows of 128 bytes
constexpr int AD_SMEM = AD_STAGES * AD_STAGE_BYTES + AD_WARPS * AD_RING * 3 * AD_ARRAY + 1024;
constexpr int AD_BLOCKS = AD_TN / 2 / AD_COLS;       // blocks of a warp in a tile: 32 rows, every other column block
constexpr uint32_t AD_IDESC = (IDESC & ~(0x3fu << 17)) | ((uint32_t)(AD_TN >> 3) << 17);
static_assert(AD_RING - 1 <= AD_BLOCKS, "blocks ahead reach the next tile at most");
static_assert(AD_STAGE_BYTES % 1024 == 0 && AD_ARRAY % 1024 == 0, "swizzle atoms must stay aligned");

struct AdamBlock {
    __nv_bfloat16 *pb, *pt;
    AdamStep step;
};

// Tiles in strips of AD_STRIP columns, columns fastest within a strip: the CTAs at work are two rows
// of tiles, 38 KB contiguous in each row of the weights, and the strip's part of B stays in L2 while
// the rows go by.  ms per step at the size above by strip width: 5 7.64, 19 7.54, 38 7.50, 76 7.46,
// 152 7.53; row tiles fastest over the whole matrix 7.66.
constexpr int AD_STRIP = 76;
__device__ __forceinline__ void adam_tile(int t, int mt, int ntl, int* mi, int* ni)
{
    const int s = t / (AD_STRIP * mt), r = t - s * AD_STRIP * mt, w = min(AD_STRIP, ntl - s * AD_STRIP);
    *mi = r / w;
    *ni = s * AD_STRIP + r - *mi * w;
}

// 4 x 4 transpose of 16-byte pieces among four neighbouring lanes: lane i's piece k becomes lane k's piece i
__device__ __forceinline__ void turn_four(uint4 (&x)[4], int lane)
{
#pragma unroll
    for (int d = 1; d <= 2; d *= 2) {
        const bool up = lane & d;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k & d) continue;
            uint4 give = up ? x[k] : x[k | d];
            give.x = __shfl_xor_sync(0xffffffffu, give.x, d);
            give.y = __shfl_xor_sync(0xffffffffu, give.y, d);
            give.z = __shfl_xor_sync(0xffffffffu, give.z, d);
            give.w = __shfl_xor_sync(0xffffffffu, give.w, d);
            if (up) x[k] = give;
            else x[k | d] = give;
        }
    }
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(src), "r"(x), "r"(y)
                 : "memory");
}

__global__ void __launch_bounds__(AD_THREADS, 1)
    gemm_adam_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                     const __grid_constant__ CUtensorMap mapP, const __grid_constant__ CUtensorMap mapM,
                     const __grid_constant__ CUtensorMap mapV, int M, int N, int nkb, int mt, int ntl, const AdamBlock w)
{
    extern __shared__ uint8_t dyn[];
    __shared__ __align__(8) uint64_t full[AD_STAGES], empty[AD_STAGES], acc_full[2], acc_empty[2], mma_done;
    __shared__ __align__(8) uint64_t arrived[AD_WARPS * AD_RING];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_issued, s_consumed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(dyn) + 1023u) & ~1023u;
    const int ntiles = mt * ntl;

    if (threadIdx.x == 0) {
        for (int s = 0; s < AD_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], AD_WARPS);  // one arrival per epilogue warp
        }
        for (int s = 0; s < AD_WARPS * AD_RING; ++s) mbar_init(&arrived[s], 1);
        mbar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_issued = 0;
        s_consumed = 0;
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(2 * AD_TN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                int mi, ni;
                adam_tile(t, mt, ntl, &mi, &ni);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % AD_STAGES;
                    if (!mbar_wait(&empty[s], ((it / AD_STAGES) & 1) ^ 1)) {
                        atomicOr(&g_tc_status, 1u);
                        ok = false;
                        break;
                    }
                    const uint32_t sa = base + s * AD_STAGE_BYTES;
                    mbar_expect_tx(&full[s], AD_STAGE_BYTES);
                    tma_load_2d(sa, &mapA, &full[s], kb * TK, mi * TM);
                    tma_load_2d(sa + A_BYTES, &mapB, &full[s], kb * TK, ni * AD_TN);
                }
            }
            s_issued = it;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0, lt = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++lt) {
                const int b = lt & 1;
                if (!mbar_wait(&acc_empty[b], ((lt >> 1) & 1) ^ 1)) {
                    atomicOr(&g_tc_status, 2u);
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * AD_TN);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % AD_STAGES;
                    if (!mbar_wait(&full[s], (it / AD_STAGES) & 1)) {
                        atomicOr(&g_tc_status, 2u);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = base + s * AD_STAGE_BYTES;
                    const uint64_t da = sw128_desc(sa), db = sw128_desc(sa + A_BYTES);
#pragma unroll
                    for (int k = 0; k < TK / UK; ++k) {
                        const uint64_t step = (uint64_t)((k * UK * 2) >> 4);
                        tc_mma(acc, da + step, db + step, AD_IDESC, (kb | k) != 0);
                    }
                    tc_commit(&empty[s]);
                }
                if (ok) tc_commit(&acc_full[b]);
            }
            s_consumed = it;
            tc_commit(&mma_done);
        }
    } else {
        // epilogue warp: TMEM lane quarter q (tile rows 32 q ..), column blocks h, h + 2 of the tile
        const int q = warp & 3, h = (warp - 2) >> 2;
        const uint32_t ring = base + AD_STAGES * AD_STAGE_BYTES + (uint32_t)(warp - 2) * (AD_RING * 3 * AD_ARRAY);
        uint64_t* const bar = arrived + (warp - 2) * AD_RING;
        const int mine = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // tiles of this CTA
        const int blocks = mine * AD_BLOCKS;
        // one lane: block j of the tile at (row, col) into place s (past the edge zeros arrive)
        auto load = [&](int s, int row, int col, int j) {
            const uint32_t dst = ring + s * 3 * AD_ARRAY;
            mbar_expect_tx(&bar[s], 3 * AD_ARRAY);
            tma_load_2d(dst, &mapP, &bar[s], col + 2 * j * AD_COLS, row);
            tma_load_2d(dst + AD_ARRAY, &mapM, &bar[s], col + 2 * j * AD_COLS, row);
            tma_load_2d(dst + 2 * AD_ARRAY, &mapV, &bar[s], col + 2 * j * AD_COLS, row);
        };
        // corner of this warp's part of tile t
        auto corner = [&](int t, int* row, int* col) {
            int mi, ni;
            adam_tile(t, mt, ntl, &mi, &ni);
            *row = mi * TM + q * 32;
            *col = ni * AD_TN + h * AD_COLS;
        };
        int row0, col_t;
        corner(blockIdx.x, &row0, &col_t);
        int issued = 0, used = 0;
        for (; issued < AD_RING - 1 && issued < blocks; ++issued)
            if (lane == 0) load(issued, row0, col_t, issued);
        bool ok = true;
        for (int lt = 0; lt < mine && ok; ++lt) {
            const int b = lt & 1;
            // one lane waits and the warp follows its result: tcgen05.ld below needs the whole warp
            int got = 0;
            if (lane == 0) got = mbar_wait(&acc_full[b], (lt >> 1) & 1) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) atomicOr(&g_tc_status, 4u);
                break;
            }
            tc_fence_after();
            int row_n = 0, col_n = 0;  // the next tile's
            if (lt + 1 < mine) corner(blockIdx.x + (lt + 1) * gridDim.x, &row_n, &col_n);
            const int row = row0 + lane;
#pragma unroll 1
            for (int j = 0; j < AD_BLOCKS; ++j, ++used) {
                const int s = used % AD_RING;
                got = mbar_wait(&bar[s], (used / AD_RING) & 1) ? 1 : 0;  // every lane: it reads what TMA wrote
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) atomicOr(&g_tc_status, 4u);
                    ok = false;
                    break;
                }
                __syncwarp();
                uint32_t r[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * AD_TN + (2 * j + h) * AD_COLS), r);
                const int col0 = col_t + 2 * j * AD_COLS;
                __nv_bfloat16* pt = w.pt + (size_t)col0 * M + row;
                uint8_t* const blk = dyn + (ring + s * 3 * AD_ARRAY - smem_u32(dyn)) + lane * 128;
                uint4 piece[4];  // the row's BF16 copy, eight columns each
#pragma unroll
                for (int c = 0; c < AD_COLS / 8; ++c) {  // eight columns at a time: two 16-byte pieces, swizzled
                    float4* const at[2] = {reinterpret_cast<float4*>(blk + 16 * ((2 * c) ^ (lane & 7))),
                                           reinterpret_cast<float4*>(blk + 16 * ((2 * c + 1) ^ (lane & 7)))};
                    constexpr int ARRAY = AD_ARRAY / 16;
                    float p[8], g[8], m[8], v[8];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        *reinterpret_cast<float4*>(p + 4 * i) = at[i][0];
                        *reinterpret_cast<float4*>(m + 4 * i) = at[i][ARRAY];
                        *reinterpret_cast<float4*>(v + 4 * i) = at[i][2 * ARRAY];
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) g[i] = __uint_as_float(r[8 * c + i]);
                    adam_many<8>(p, g, m, v, w.step);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        at[i][0] = *reinterpret_cast<const float4*>(p + 4 * i);
                        at[i][ARRAY] = *reinterpret_cast<const float4*>(m + 4 * i);
                        at[i][2 * ARRAY] = *reinterpret_cast<const float4*>(v + 4 * i);
                    }
                    const int col = col0 + 8 * c;
                    const uint2 lo = pack_bf16x4(make_float4(p[0], p[1], p[2], p[3])),
                                hi = pack_bf16x4(make_float4(p[4], p[5], p[6], p[7]));
                    piece[c] = make_uint4(lo.x, lo.y, hi.x, hi.y);
                    if (row < M && col < N) {  // N is a multiple of 8
                        const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&piece[c]);
#pragma unroll
                        for (int k = 0; k < 8; ++k, pt += M) *pt = e[k];
                    }
                    if (c == 0) {
                        // the other place is free once the block before has been read from it
                        if (lane == 0 && issued < blocks) {
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                            const int ahead = j + AD_RING - 1;  // blocks into this tile, or the next
                            if (ahead < AD_BLOCKS) load(issued % AD_RING, row0, col_t, ahead);
                            else load(issued % AD_RING, row_n, col_n, ahead - AD_BLOCKS);
                        }
                        if (issued < blocks) ++issued;
                    }
                }
                // the row-major copy, turned around among four lanes: a store covers 64 bytes of eight rows
                // (pieces of 16 bytes a row at a time would write half sectors)
                turn_four(piece, lane);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int rr = row0 + (lane & ~3) + k, col = col0 + 8 * (lane & 3);
                    if (rr < M && col < N) *reinterpret_cast<uint4*>(w.pb + (size_t)rr * N + col) = piece[k];
                }
                // the block leaves; the place of the one before is free once it has been read
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    if (row0 < M && col0 < N) {
                        const uint32_t src = ring + s * 3 * AD_ARRAY;
                        tma_store_2d(&mapP, src, col0, row0);
                        tma_store_2d(&mapM, src + AD_ARRAY, col0, row0);
                        tma_store_2d(&mapV, src + 2 * AD_ARRAY, col0, row0);
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                if (j == AD_BLOCKS - 1) {  // every tcgen05.ld of this warp has completed: hand the accumulator back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[b]);
                }
            }
            row0 = row_n;
            col_t = col_n;
        }
        if (lane == 0) {
            // blocks that were asked for and not used (only after a wait gave up) must land before the CTA
            // exits, and the last ones must have left shared memory
            for (; used < issued; ++used)
                if (!mbar_wait(&bar[used % AD_RING], (used / AD_RING) & 1)) {
                    atomicOr(&g_tc_status, 16u);
                    break;
                }
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_wait(&mma_done, 0)) atomicOr(&g_tc_status, 8u);
        for (int it = s_consumed; it < s_issued; ++it)
            if (!mbar_wait(&full[it % AD_STAGES], (it / AD_STAGES) & 1)) {
                atomicOr(&g_tc_status, 16u);
                break;
            }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * AD_TN) : "memory");
    }
}

}  // namespace

// gemm_tc_kernel on `grid` CTAs, in clusters of CL
template <int CL, bool PROBE = false, class... Args>
static cudaError_t launch_gemm(unsigned grid, cudaStream_t st, Args... args)
{
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<CL, PROBE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<CL, PROBE>, args...);
}

cudaError_t gemm_bf16_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb,
                         float* C, int ldc, float alpha, float beta, int split_k, cudaStream_t st,
                         const float* alpha4, int span)
{
    if (alpha4 && (span < 1 || (long long)4 * span < N)) return cudaErrorInvalidValue;
    const float4 av = alpha4 ? make_float4(alpha4[0], alpha4[1], alpha4[2], alpha4[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return cudaErrorInvalidValue;
    if (lda % 8 || ldb % 8 || lda < K || ldb < K || ldc < N) return cudaErrorInvalidValue;
    EncodeTiled fn = encode_tiled();
    if (!fn) return cudaErrorNotSupported;
    const int nkb = (K + TK - 1) / TK;
    if (split_k < 1) split_k = 1;
    if (split_k > nkb) split_k = nkb;
    const int kb_per = (nkb + split_k - 1) / split_k;
    split_k = (nkb + kb_per - 1) / kb_per;  // no empty slice
    const int mt = (M + TM - 1) / TM, ntl = (N + TN - 1) / TN;
    const long long ntiles = (long long)mt * ntl * split_k;
    if (ntiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool pair = mt % 2 == 0 && kb_per >= PAIR_MIN_K && ntiles * kb_per >= (long long)PAIR_MIN_WORK * sms;
    alignas(64) CUtensorMap mapA, mapB;
    if (!make_map(fn, &mapA, A, M, K, lda, TM) || !make_map(fn, &mapB, B, N, K, ldb, pair ? TN / 2 : TN))
        return cudaErrorInvalidValue;
    if (split_k > 1 && beta != 1.f && (e = scale_f32(C, M, N, ldc, beta, st)) != cudaSuccess) return e;
    const unsigned grid = (unsigned)(ntiles < sms ? ntiles : (pair ? sms / 2 * 2 : sms));
    const int atomic = split_k > 1 ? 1 : 0, sp = alpha4 ? span : 0;
    return pair ? launch_gemm<2>(grid, st, mapA, mapB, M, N, nkb, kb_per, mt, ntl, (int)ntiles, C, ldc, alpha, beta, atomic, av, sp)
                : launch_gemm<1>(grid, st, mapA, mapB, M, N, nkb, kb_per, mt, ntl, (int)ntiles, C, ldc, alpha, beta, atomic, av, sp);
}

// a row-major FP32 [rows][cols] array in blocks of 32 x AD_COLS, 128-byte swizzle
static bool make_map_f32(EncodeTiled fn, CUtensorMap* map, float* ptr, int rows, int cols)
{
    const cuuint64_t dim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t stride[1] = {(cuuint64_t)cols * 4};
    const cuuint32_t box[2] = {(cuuint32_t)AD_COLS, 32u};
    const cuuint32_t estride[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, ptr, dim, stride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

cudaError_t gemm_adam_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, float* p,
                         float* m, float* v, float lr, float b1, float b2, float eps, int t, __nv_bfloat16* pb,
                         __nv_bfloat16* pt, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0 || N % 8) return cudaErrorInvalidValue;
    const uintptr_t al = reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v) |
                         reinterpret_cast<uintptr_t>(pb) | reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B);
    if (al & 15) return cudaErrorInvalidValue;
    if (lda % 8 || ldb % 8 || lda < K || ldb < K) return cudaErrorInvalidValue;
    EncodeTiled fn = encode_tiled();
    if (!fn) return cudaErrorNotSupported;
    alignas(64) CUtensorMap mapA, mapB, mapP, mapM, mapV;
    if (!make_map(fn, &mapA, A, M, K, lda, TM) || !make_map(fn, &mapB, B, N, K, ldb, AD_TN) ||
        !make_map_f32(fn, &mapP, p, M, N) || !make_map_f32(fn, &mapM, m, M, N) || !make_map_f32(fn, &mapV, v, M, N))
        return cudaErrorInvalidValue;
    const int mt = (M + TM - 1) / TM;
    const long long ntiles = (long long)mt * ((N + AD_TN - 1) / AD_TN);
    if (ntiles > 0x7fffffffLL - 4096) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_adam_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AD_SMEM);
    if (e != cudaSuccess) return e;
    const AdamBlock w = {pb, pt, adam_step(lr, b1, b2, eps, t)};
    const long long grid = ntiles < sms ? ntiles : sms;
    gemm_adam_kernel<<<(unsigned)grid, AD_THREADS, AD_SMEM, st>>>(mapA, mapB, mapP, mapM, mapV, M, N, (K + TK - 1) / TK, mt, (N + AD_TN - 1) / AD_TN, w);
    return cudaGetLastError();
}

cudaError_t gemm_wait_probe(double seconds, cudaStream_t st)
{
    if (!(seconds > 0.0) || seconds > 2.0) return cudaErrorInvalidValue;
    wait_probe_kernel<<<1, 32, 0, st>>>((unsigned long long)(seconds * 1e9));
    return cudaGetLastError();
}

cudaError_t gemm_pair_probe(int rank, int stage, unsigned* status, cudaStream_t st)
{
    constexpr int K = 20 * TK;
    if (rank < 0 || rank > 1 || stage < 0 || stage >= 20) return cudaErrorInvalidValue;
    EncodeTiled fn = encode_tiled();
    if (!fn) return cudaErrorNotSupported;
    const size_t ab = (size_t)2 * TM * K * sizeof(__nv_bfloat16), c = (size_t)2 * TM * TN * sizeof(float);
    char* mem = nullptr;
    cudaError_t e = cudaMalloc(&mem, 2 * ab + c);
    if (e != cudaSuccess) return e;
    alignas(64) CUtensorMap mapA, mapB;
    const __nv_bfloat16 *A = reinterpret_cast<__nv_bfloat16*>(mem), *B = reinterpret_cast<__nv_bfloat16*>(mem + ab);
    if (!make_map(fn, &mapA, A, 2 * TM, K, K, TM) || !make_map(fn, &mapB, B, TN, K, K, TN / 2)) e = cudaErrorInvalidValue;
    if (e == cudaSuccess) e = cudaMemsetAsync(mem, 0, 2 * ab + c, st);
    if (e == cudaSuccess)
        e = launch_gemm<2, true>(2, st, mapA, mapB, 2 * TM, TN, 20, 20, 2, 1, 2, reinterpret_cast<float*>(mem + 2 * ab), TN, 1.f,
                                 0.f, 0, make_float4(0.f, 0.f, 0.f, 0.f), 2 * stage + rank);
    const cudaError_t e2 = cudaStreamSynchronize(st);
    cudaFree(mem);
    if (e == cudaSuccess) e = e2;
    return e == cudaSuccess ? cudaMemcpyFromSymbol(status, g_tc_status, sizeof *status) : e;
}

cudaError_t gemm_tc_status(unsigned* status)
{
    unsigned v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_status, sizeof v);
    if (e != cudaSuccess) return e;
    *status = v;
    if (v) {
        const unsigned zero = 0;
        e = cudaMemcpyToSymbol(g_tc_status, &zero, sizeof zero);
    }
    return e;
}

}  // namespace es
