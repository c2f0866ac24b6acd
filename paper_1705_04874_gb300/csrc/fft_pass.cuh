// Fused pseudo-spectral derivative passes (Sec. II-A of Das, Chen & Hobson,
// arXiv 1705.04874: Fourier-domain spatial derivatives on a staggered grid).
//
// One CTA owns a tile of 32 real pencils along the pass axis, packed two at a
// time into 16 complex lines (line c = pencil 2c + i * pencil 2c+1; y and z
// passes with an odd nx: pencil c + i * pencil 16+c).  For
// each job it runs: near stencil -> forward FFT along the axis -> multiply by
// (H - H_near) / n -> inverse FFT -> field-update epilogue.  Because the
// multiplier is Hermitian (a real field has a real derivative, including at
// the Nyquist bin, where it is the real number -/+ pi / d), the real and
// imaginary parts of the result are the derivatives of the two packed pencils.
//
// The transform of length n = RA * RB is a two-stage Stockham autosort FFT
// (radix RA with stride n/RA, then radix RB with twiddles exp(-2 pi i k r / n)).
// Its last forward stage leaves each thread holding exactly the elements
// b + q n/RB that the first stage of the inverse (run as a forward transform
// of the conjugate, with the radices in reverse order) needs, so the
// multiply and that stage happen in registers; shared memory is touched only
// between stages.  The inverse's last stage ends on the same elements the
// first forward stage loaded, so the epilogue writes where the loads read.
// Three-stage plans (Core3: 125 = 5 x 5 x 5, 75 = 3 x 5 x 5) run their middle
// stages through shared memory and keep the same first / last-stage layout.
//
// Near part.  Each derivative is a near part plus a far part (es_internal.h):
// the multiplier tables hold H_far / n, and the NEAR_TAPS-point stencil is
// formed first, from the staged source tile, several consecutive positions per
// thread with the window sliding through registers (1 + 9 / 16 shared loads
// per output along y and z instead of 10).  It waits in tensor memory, which
// nothing else here uses, until the inverse transform is done.  In exact
// arithmetic the sum is the spectral derivative itself; in FP32 the FFT's
// roundoff, which is spread over the whole pencil, is scaled down by
// |H_far| / |H| (about 1 %), so far-away receivers no longer see the FP32
// noise of the pencil's largest values.
//
// The passes (but for the y and z passes of the shortest and the odd lengths,
// pass_strided_once) are persistent: while a CTA works on one tile, the next one's
// source arrives in shared memory (cp.async), so that the 3 CTAs an SM holds at
// n = 256 (72 KB each) have 6 tiles in hand.  What bounds them is memory: at
// 256^3 (one GB300, 6.68 TB/s copy rate) the y / z velocity passes move 844 MB
// in 0.158 / 0.163 ms (5.3 TB/s), the stress passes 1.21 GB in 0.213 / 0.217 ms
// (5.7 TB/s), the x passes the same bytes in 0.182 and 0.227 ms.  One tile per
// CTA (four CTAs per SM, the source read straight into registers and fetched
// again from L2 for the stencil) took 0.188 / 0.203, 0.245 / 0.258, 0.191 and
// 0.242 ms: a chain of load, transform, reload and update with nothing to
// overlap it but the other CTAs.  Tried on the way and dropped: four pencils
// per thread (half the instructions, 12 warps per SM: 0.191 ms, latency-bound);
// the near parts in a third shared tile and one tile per CTA (0.188 ms); slab
// rows left to the warps that own them (0.231 ms, the others wait).
//
// Strided passes (y, z): a tile is 32 consecutive x (128-byte rows) by the
// whole pencil.  The x pass stages 32 whole x-lines (contiguous in memory),
// turns them around into the same [position][pencil] rows, and reads the far
// parts back from there line by line.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <algorithm>
#include <type_traits>
#include <utility>

#include "es_internal.h"

namespace es {

// ---------------------------------------------------------------------------
// compile-time twiddles W_R^M = exp(-2 pi i M / R)
// ---------------------------------------------------------------------------
__host__ __device__ constexpr double ce_cos_frac(long m, long r)
{
    // cos(2 pi m / r): exact at multiples of pi / 2, Taylor series otherwise
    long mm = ((m % r) + r) % r;
    if ((4 * mm) % r == 0) {
        long q = (4 * mm) / r;
        return q == 0 ? 1.0 : (q == 2 ? -1.0 : 0.0);
    }
    double x = 6.283185307179586476925286766559 * (double)mm / (double)r;
    if (2 * mm > r) x -= 6.283185307179586476925286766559;
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 40; ++k) {
        term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double ce_sin_frac(long m, long r)
{
    return ce_cos_frac(4 * m - r, 4 * r);  // sin(t) = cos(t - pi/2)
}

template <int... Is, class F>
__device__ __forceinline__ void sfor_impl(std::integer_sequence<int, Is...>, F&& f)
{
    (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f)
{
    sfor_impl(std::make_integer_sequence<int, N>{}, f);
}

// Packed FP32 pairs (PTX f32x2): two operations in one instruction, each
// component rounded exactly as the scalar operation
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\n"
        "add.rn.f32x2 rd, ra, rb;\nmov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 d;
    asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\n"
        "sub.rn.f32x2 rd, ra, rb;\nmov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\n"
        "mul.rn.f32x2 rd, ra, rb;\nmov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n.reg .b64 ra, rb, rc, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmov.b64 rc, {%6, %7};\n"
        "fma.rn.f32x2 rd, ra, rb, rc;\nmov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 rep2(float s) { return make_float2(s, s); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return sub2(a, b); }
// a - i b and a + i b
__device__ __forceinline__ float2 csub_i(float2 a, float2 b)
{
    return make_float2(__fadd_rn(a.x, b.y), __fsub_rn(a.y, b.x));
}
__device__ __forceinline__ float2 cadd_i(float2 a, float2 b)
{
    return make_float2(__fsub_rn(a.x, b.y), __fadd_rn(a.y, b.x));
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// v W_R^M, a compile-time constant
template <int R, int M>
__device__ __forceinline__ float2 twc(float2 v)
{
    constexpr int mm = ((M % R) + R) % R;
    if constexpr (mm == 0) {
        return v;
    } else if constexpr ((4 * mm) % R == 0) {
        constexpr int q = (4 * mm) / R;  // rotation by -i q
        if constexpr (q == 1) return make_float2(v.y, -v.x);
        else if constexpr (q == 2) return make_float2(-v.x, -v.y);
        else return make_float2(-v.y, v.x);
    } else {
        constexpr float c = (float)ce_cos_frac(mm, R);
        constexpr float s = (float)(-ce_sin_frac(mm, R));
        return make_float2(c * v.x - s * v.y, c * v.y + s * v.x);
    }
}

// Index check of the bounds-checked build (ES_BOUNDS, es_internal.h): true
// when 0 <= i < n; otherwise the first such index is recorded with the source
// line and the caller skips the access.  Always true in the release build.
__device__ __forceinline__ bool inb(unsigned long long* bad, long long i, long long n, int line)
{
#if ES_BOUNDS
    if (i >= 0 && i < n) return true;
    if (bad) atomicCAS(bad, 0ull, ((unsigned long long)line << 40) | ((unsigned long long)i & 0xFFFFFFFFFFull));
    return false;
#else
    (void)bad;
    (void)i;
    (void)n;
    (void)line;
    return true;
#endif
}
#define ES_INB(p, i, n) inb((p).bad, (long long)(i), (long long)(n), __LINE__)

// ---------------------------------------------------------------------------
// forward DFTs of small sizes in registers: a[k] <- sum_j a[j] W_R^(jk)
// ---------------------------------------------------------------------------
template <int R> struct Dft;

template <> struct Dft<2> {
    static __device__ __forceinline__ void run(float2* a)
    {
        float2 t = a[0];
        a[0] = cadd(t, a[1]);
        a[1] = csub(t, a[1]);
    }
};

template <> struct Dft<3> {
    static __device__ __forceinline__ void run(float2* a)
    {
        constexpr float h = 0.86602540378443864676f;  // sqrt(3) / 2
        float2 t1 = cadd(a[1], a[2]), t2 = csub(a[1], a[2]);
        float2 m = make_float2(a[0].x - 0.5f * t1.x, a[0].y - 0.5f * t1.y);
        a[0] = cadd(a[0], t1);
        a[1] = make_float2(m.x + h * t2.y, m.y - h * t2.x);  // m - i h t2
        a[2] = make_float2(m.x - h * t2.y, m.y + h * t2.x);  // m + i h t2
    }
};

template <> struct Dft<4> {
    static __device__ __forceinline__ void run(float2* a)
    {
        float2 s02 = cadd(a[0], a[2]), d02 = csub(a[0], a[2]);
        float2 s13 = cadd(a[1], a[3]), d13 = csub(a[1], a[3]);
        a[0] = cadd(s02, s13);
        a[2] = csub(s02, s13);
        a[1] = csub_i(d02, d13);
        a[3] = cadd_i(d02, d13);
    }
};

template <> struct Dft<5> {
    static __device__ __forceinline__ void run(float2* a)
    {
        constexpr float c1 = 0.30901699437494742410f;   // cos(2 pi / 5)
        constexpr float c2 = -0.80901699437494742410f;  // cos(4 pi / 5)
        constexpr float s1 = 0.95105651629515357212f;   // sin(2 pi / 5)
        constexpr float s2 = 0.58778525229247312917f;   // sin(4 pi / 5)
        float2 t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]);
        float2 t3 = csub(a[1], a[4]), t4 = csub(a[2], a[3]);
        float2 b1 = make_float2(a[0].x + c1 * t1.x + c2 * t2.x, a[0].y + c1 * t1.y + c2 * t2.y);
        float2 b2 = make_float2(a[0].x + c2 * t1.x + c1 * t2.x, a[0].y + c2 * t1.y + c1 * t2.y);
        float2 e1 = make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y);
        float2 e2 = make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y);
        a[0] = cadd(a[0], cadd(t1, t2));
        a[1] = csub_i(b1, e1);
        a[4] = cadd_i(b1, e1);
        a[2] = csub_i(b2, e2);
        a[3] = cadd_i(b2, e2);
    }
};

// Composite R = P * Q in registers (Cooley-Tukey):
// X[k1 + P k2] = sum_n2 W_Q^(n2 k2) W_R^(n2 k1) sum_n1 a[Q n1 + n2] W_P^(n1 k1)
template <int P, int Q> struct DftPQ {
    static __device__ __forceinline__ void run(float2* a)
    {
        constexpr int R = P * Q;
        float2 B[Q][P];
        sfor<Q>([&](auto n2) {
            float2 v[P];
            sfor<P>([&](auto n1) { v[n1] = a[Q * n1 + n2]; });
            Dft<P>::run(v);
            sfor<P>([&](auto k1) { B[n2][k1] = twc<R, decltype(n2)::value * decltype(k1)::value>(v[k1]); });
        });
        sfor<P>([&](auto k1) {
            float2 v[Q];
            sfor<Q>([&](auto n2) { v[n2] = B[n2][k1]; });
            Dft<Q>::run(v);
            sfor<Q>([&](auto k2) { a[k1 + P * k2] = v[k2]; });
        });
    }
};
template <> struct Dft<6> : DftPQ<2, 3> {};
template <> struct Dft<8> : DftPQ<2, 4> {};
template <> struct Dft<10> : DftPQ<2, 5> {};
template <> struct Dft<12> : DftPQ<4, 3> {};
template <> struct Dft<15> : DftPQ<3, 5> {};
template <> struct Dft<16> : DftPQ<4, 4> {};
template <> struct Dft<25> : DftPQ<5, 5> {};

// ---------------------------------------------------------------------------
// epilogues
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool in_slab(int pos, int n, int L)
{
    return L > 0 && (pos < L || pos >= n - 1 - L);
}

// index of (x, y, z) in the slab array of `axis` (slab coordinate sp)
__device__ __forceinline__ size_t slab_index(int axis, int x, int y, int z, int sp, int nx, int ny, int S)
{
    if (axis == 0) return (size_t)sp + (size_t)S * ((size_t)y + (size_t)ny * z);
    if (axis == 1) return (size_t)x + (size_t)nx * ((size_t)sp + (size_t)S * z);
    return (size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * sp);
}

// Split-field update inside a PML slab: s <- P (P s + inc).  Returns the
// change of the split, which is the change of the field total.  The epilogues
// spell out their roundings (__fmaf_rn / __fmul_rn / __fadd_rn) so that every
// kernel that updates a field does so in the same FP32 operations, whatever
// the compiler would contract around them.
__device__ __forceinline__ float split_delta(float* slab, size_t si, float P, float inc)
{
    const float s = slab[si];
    const float sn = __fmul_rn(P, __fmaf_rn(P, s, inc));
    slab[si] = sn;
    return __fsub_rn(sn, s);
}
// dt c D, rounded after each product
__device__ __forceinline__ float increment(float dt, float c, float d) { return __fmul_rn(__fmul_rn(dt, c), d); }
// lambda + 2 mu (diag) or lambda
__device__ __forceinline__ float normal_coef(float lam, float mu, bool diag) { return diag ? __fmaf_rn(2.f, mu, lam) : lam; }

// Field totals take their increment by a vector reduction in L2 (atomicAdd
// with the result unused): within one pass every total receives exactly one
// increment, and passes are stream-ordered, so the result is the plain
// rounded sum, deterministic, while the epilogue never waits for the old
// value.
// ---- y / z epilogue: two cells per thread and position ----
// A thread's pencil pair is x0 + 2c, x0 + 2c + 1 with an even nx (V = 2: 8-byte
// accesses); with an odd one, whose rows start anywhere, x0 + c and x0 + D + c
// (V = 1, D pairs per row: two 4-byte accesses, each coalesced over the row's
// half).  two: whether the second cell exists (V = 1; V = 2 has both).
template <int V, int D>
__device__ __forceinline__ float2 ld_pair(const float* q, bool two)
{
    if constexpr (V == 2) return *reinterpret_cast<const float2*>(q);
    return make_float2(q[0], two ? q[D] : 0.f);
}
// the same from memory no kernel writes (the coefficients)
template <int V, int D>
__device__ __forceinline__ float2 ldg_pair(const float* q, bool two)
{
    if constexpr (V == 2) return __ldg(reinterpret_cast<const float2*>(q));
    return make_float2(__ldg(q), two ? __ldg(q + D) : 0.f);
}
template <int V, int D>
__device__ __forceinline__ void st_pair(float* q, float2 v, bool two)
{
    if constexpr (V == 2) {
        *reinterpret_cast<float2*>(q) = v;
    } else {
        q[0] = v.x;
        if (two) q[D] = v.y;
    }
}
template <int V, int D>
__device__ __forceinline__ void red_pair(float* q, float2 v, bool two)
{
    if constexpr (V == 2) {
        atomicAdd(reinterpret_cast<float2*>(q), v);
    } else {
        atomicAdd(q, v.x);
        if (two) atomicAdd(q + D, v.y);
    }
}

// Epilogue for one cell (what is left of an x pass's tile past its whole quads, or
// all of it where its arrays are not on 16-byte boundaries; the circulant passes):
// the same arithmetic as the pass epilogues, one cell at a time.
__device__ __forceinline__ void epilogue_one(const PassParams& p, const PassJob& J, size_t q, int pos, int x, int y,
                                             int z, float d, size_t off, size_t soff)
{
    if (!ES_INB(p, off + q, p.ext_f)) return;
    if (J.kind == JOB_STORE) {
        J.tgt[0][off + q] = d;
        return;
    }
    if (!ES_INB(p, q, p.ext_c)) return;
    const float dt = p.dt;
    const bool slab = in_slab(pos, p.n, p.L);
    const int S = p.S;
    if (J.kind == JOB_SINGLE) {
        float inc = increment(dt, __ldg(J.coef[0] + q), d);
        if (slab) {
            const float P = __ldg((J.stag ? p.ps : p.pc) + pos);
            const size_t si = slab_index(p.axis, x, y, z, slab_pos(pos, p.n, p.L, p.S), p.nx, p.ny, S);
            if (!ES_INB(p, soff + si, p.ext_s)) return;
            inc = split_delta(J.slab[0], soff + si, P, inc);
        }
        atomicAdd(J.tgt[0] + off + q, inc);
    } else {
        const float lam = __ldg(J.coef[0] + q), mu = __ldg(J.coef[1] + q);
        const float P = slab ? __ldg(p.pc + pos) : 1.f;
        const size_t si = slab ? slab_index(p.axis, x, y, z, slab_pos(pos, p.n, p.L, p.S), p.nx, p.ny, S) : 0;
        if (slab && !ES_INB(p, soff + si, p.ext_s)) return;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            float inc = increment(dt, normal_coef(lam, mu, t == J.diag), d);
            if (slab) inc = split_delta(J.slab[t], soff + si, P, inc);
            atomicAdd(J.tgt[t] + off + q, inc);
        }
    }
}

// ---------------------------------------------------------------------------
// FFT core on the shared [pos][quad] rows (one buffer, updated in place:
// every stage reads all its inputs, the block synchronises, then it writes).
// Thread (j, c): j = tid / PAIRS, quad c = tid % PAIRS.
// ---------------------------------------------------------------------------
constexpr int PAIRS = 16;  // pencil pairs per row of a tile (32 pencils, 128 bytes)

// the butterfly of a stage of B dealt over T threads: past the last one the last
// one again (the same values go to the same places, which costs less than
// branches around register arrays: those spill)
template <int B, int T>
__device__ __forceinline__ int butterfly(int b)
{
    return B % T == 0 ? b : min(b, B - 1);
}

template <int RA, int RB, int T_, int PR = PAIRS>
struct Core {
    static constexpr int N = RA * RB;
    static constexpr int R1 = RA;
    static constexpr int BA = N / RA;   // stage-A butterflies
    static constexpr int BB = N / RB;   // stage-B butterflies
    static constexpr int T = T_;        // threads per pair
    static constexpr int MA = (BA + T - 1) / T, MB = (BB + T - 1) / T;  // butterflies per thread

    // first forward stage (radix RA, Stockham Ns = 1) on elements b + r BA, b = j + m T; row(e)
    // reads source element e
    template <class Row>
    static __device__ __forceinline__ void stageA(float2 (&a)[MA][RA], int j, Row row)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
            const int b = butterfly<BA, T>(j + m * T);
#pragma unroll
            for (int r = 0; r < RA; ++r) a[m][r] = row(b + r * BA);
            Dft<RA>::run(a[m]);
        }
    }
    // its results to elements b RA + q
    static __device__ __forceinline__ void stageA_store(const float2 (&a)[MA][RA], float2* buf, int j, int c)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
            const int b = butterfly<BA, T>(j + m * T);
#pragma unroll
            for (int q = 0; q < RA; ++q) buf[(b * RA + q) * PR + c] = a[m][q];
        }
    }

    // stage B (radix RB, Ns = RA), spectral multiply, conjugate, first inverse
    // stage (radix RB, Ns = 1), all in registers
    static __device__ __forceinline__ void middle(float2* buf, const float2* tw, const float2* H, int j, int c)
    {
        float2 v[MB][RB];
#pragma unroll
        for (int m = 0; m < MB; ++m) {
            const int b = butterfly<BB, T>(j + m * T);
            const int k = b % RA;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const float2 x = buf[(b + r * BB) * PR + c];
                v[m][r] = r == 0 ? x : cmul(x, tw[k * r]);
            }
            Dft<RB>::run(v[m]);
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                const float2 y = cmul(H[b + q * BB], v[m][q]);
                v[m][q] = make_float2(y.x, -y.y);
            }
            Dft<RB>::run(v[m]);
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < MB; ++m) {
            const int b = butterfly<BB, T>(j + m * T);
#pragma unroll
            for (int q = 0; q < RB; ++q) buf[(b * RB + q) * PR + c] = v[m][q];
        }
    }

    // last inverse stage (radix RA, Ns = RB): conj(a[m][q]) = the result at
    // element b + q BA
    static __device__ __forceinline__ void stageA_inv(const float2* buf, const float2* tw, float2 (&a)[MA][RA], int j,
                                                      int c)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
            const int b = butterfly<BA, T>(j + m * T);
            const int k = b % RB;
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                const float2 x = buf[(b + r * BA) * PR + c];
                a[m][r] = r == 0 ? x : cmul(x, tw[k * r]);
            }
            Dft<RA>::run(a[m]);
        }
    }
    // put(e, v) for every element e this thread's last stage ends on
    template <class Put>
    static __device__ __forceinline__ void results(const float2 (&a)[MA][RA], int j, Put put)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
            const int b = butterfly<BA, T>(j + m * T);
#pragma unroll
            for (int q = 0; q < RA; ++q) put(b + q * BA, a[m][q]);
        }
    }
};

// Three-stage plan n = R1 R2 R3 (Stockham, as Core): forward stages of radix
// R1, R2, R3, the spectral multiply on the elements the last one leaves in a
// thread's registers, then the inverse (forward DFTs of the conjugate) with
// the radices reversed: R3 on those same elements, R2, and R1, which ends on
// the elements j + q n/R1 the first stage read.  A stage of radix R after
// stages whose radices multiply to Ns: butterfly b (k = b mod Ns) reads
// elements b + r n/R times W_(Ns R)^(k r), runs the R-point DFT and writes
// element (b / Ns) Ns R + k + q Ns.  All stages but the first and the last
// run on the shared buffer, every butterfly of a stage by one thread.
template <int R1_, int R2, int R3, int T_, int PR = PAIRS>
struct Core3 {
    static constexpr int R1 = R1_;
    static constexpr int N = R1 * R2 * R3;
    static constexpr int BA = N / R1;  // first / last stage butterflies
    static constexpr int T = T_;       // threads per pair
    static constexpr int MA = BA / T;  // first / last stage butterflies per thread
    static_assert(BA % T == 0, "the first stage deals its butterflies evenly");
    template <class Row>
    static __device__ __forceinline__ void stageA(float2 (&a)[MA][R1], int j, Row row)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
#pragma unroll
            for (int r = 0; r < R1; ++r) a[m][r] = row(j + m * T + r * BA);
            Dft<R1>::run(a[m]);
        }
    }
    static __device__ __forceinline__ void stageA_store(const float2 (&a)[MA][R1], float2* buf, int j, int c)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m)
#pragma unroll
            for (int q = 0; q < R1; ++q) buf[((j + m * T) * R1 + q) * PR + c] = a[m][q];
    }

    // one stage of radix R after radices multiplying to NS, shared buffer to
    // shared buffer (reads, block barrier, writes)
    template <int R, int NS>
    static __device__ __forceinline__ void stage(float2* buf, const float2* tw, int j, int c)
    {
        constexpr int B = N / R, M = (B + T - 1) / T, TS = N / (NS * R);
        float2 v[M][R];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int b = butterfly<B, T>(j + m * T);
            const int k = b % NS;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 x = buf[(b + r * B) * PR + c];
                v[m][r] = r == 0 ? x : cmul(x, tw[k * r * TS]);
            }
            Dft<R>::run(v[m]);
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int b = butterfly<B, T>(j + m * T);
            const int k = b % NS, o = (b / NS) * NS * R + k;
#pragma unroll
            for (int q = 0; q < R; ++q) buf[(o + q * NS) * PR + c] = v[m][q];
        }
    }

    static __device__ __forceinline__ void middle(float2* buf, const float2* tw, const float2* H, int j, int c)
    {
        stage<R2, R1>(buf, tw, j, c);
        __syncthreads();
        {
            // last forward stage (radix R3, Ns = n/R3, so k = b), multiply,
            // conjugate, first inverse stage (radix R3, Ns = 1) in registers
            constexpr int B = N / R3, M = (B + T - 1) / T;
            float2 v[M][R3];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int b = butterfly<B, T>(j + m * T);
#pragma unroll
                for (int r = 0; r < R3; ++r) {
                    const float2 x = buf[(b + r * B) * PR + c];
                    v[m][r] = r == 0 ? x : cmul(x, tw[b * r]);
                }
                Dft<R3>::run(v[m]);
#pragma unroll
                for (int q = 0; q < R3; ++q) {
                    const float2 y = cmul(H[b + q * B], v[m][q]);
                    v[m][q] = make_float2(y.x, -y.y);
                }
                Dft<R3>::run(v[m]);
            }
            __syncthreads();
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int b = butterfly<B, T>(j + m * T);
#pragma unroll
                for (int q = 0; q < R3; ++q) buf[(b * R3 + q) * PR + c] = v[m][q];
            }
        }
        __syncthreads();
        stage<R2, R3>(buf, tw, j, c);
    }

    // last inverse stage (radix R1, Ns = n/R1, so k = b): conj(a[m][q]) = the
    // result at element b + q BA, b = j + m T
    static __device__ __forceinline__ void stageA_inv(const float2* buf, const float2* tw, float2 (&a)[MA][R1], int j,
                                                      int c)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m) {
            const int b = j + m * T;
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const float2 x = buf[(b + r * BA) * PR + c];
                a[m][r] = r == 0 ? x : cmul(x, tw[b * r]);
            }
            Dft<R1>::run(a[m]);
        }
    }
    template <class Put>
    static __device__ __forceinline__ void results(const float2 (&a)[MA][R1], int j, Put put)
    {
#pragma unroll
        for (int m = 0; m < MA; ++m)
#pragma unroll
            for (int q = 0; q < R1; ++q) put(j + m * T + q * BA, a[m][q]);
    }
};

// the FFT core of a plan (RC = 1: two stages)
template <int RA, int RB, int RC, int T, int PR = PAIRS>
using CoreOf = std::conditional_t<RC == 1, Core<RA, RB, T, PR>, Core3<RA, RB, RC, T, PR>>;

// asynchronous BYTES-byte global -> shared copy (cp.async); ok == false writes
// zeros and reads nothing
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool ok)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = ok ? BYTES : 0;
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(n)
                     : "memory");
}
__device__ __forceinline__ void cp_async_commit_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
}

template <int T>
__host__ __device__ constexpr int pass_threads() { return T * PAIRS; }

// blocks per SM the register budget is sized for, from the pairs a thread
// carries through its largest stage (80 registers up to 16 pairs: measured on
// the two-stage plans, where a spill costs more than the CTA it buys)
template <int RA, int RB, int RC, int T>
__host__ __device__ constexpr int pass_min_blocks(int small = 1024)
{
    constexpr int N = RA * RB * RC;
    auto held = [](int r) { return (N / r + T - 1) / T * r; };
    constexpr int top = held(RA) > held(RB) ? (held(RA) > held(RC) ? held(RA) : held(RC))
                                            : (held(RB) > held(RC) || RC == 1 ? held(RB) : held(RC));
    // `small`: threads per SM for plans that hold 10 pairs or fewer
    const int per_sm = top > 16 ? 640 : (top > 10 ? 768 : small);
    const int b = per_sm / ((pass_threads<T>() + 31) / 32 * 32);
    return b < 1 ? 1 : (b > 24 ? 24 : b);
}

// Whether the near parts wait in tensor memory (2 n / T columns of 32 bits per
// warp) instead of a third shared tile: from 12 positions per thread on, three
// tiles per CTA, not the registers, would limit the CTAs on an SM.  tcgen05.st /
// ld work on whole warps, four of them side by side in the tensor memory's lanes.
template <int N, int T>
__host__ __device__ constexpr bool near_in_tmem()
{
    return N / T >= 12 && N / T % 4 == 0 && pass_threads<T>() % 32 == 0;
}
// columns to allocate: a power of two, at least 32
template <int N, int T>
__host__ __device__ constexpr unsigned tmem_columns()
{
    constexpr unsigned n = 2 * (N / T) * ((pass_threads<T>() / 32 + 3) / 4);
    return n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : 256));
}
// positions whose near parts move to or from tensor memory (and whose
// coefficients are in flight) at once
template <int RN>
__host__ __device__ constexpr int epi_batch()
{
    static_assert(RN % 4 == 0 || RN % 5 == 0, "whole batches");
    return RN % 4 == 0 ? 4 : 5;
}

// shared bytes of the y / z passes: two tiles [N][PAIRS] (the current one,
// source then FFT buffer; the next one, arriving), the near parts where they
// are not in tensor memory, twiddles and both multipliers
template <int N, int T>
__host__ __device__ constexpr size_t pass_smem_strided()
{
    return (near_in_tmem<N, T>() ? 2 : 3) * sizeof(float2) * N * PAIRS + 3 * sizeof(float2) * N;
}
// of the x pass: the same (the tile as it is in memory, the next one's place,
// and its turned-around rows); lengths that are not a multiple of 16: the
// rows, the near parts, twiddles and multiplier
template <int N, int T>
__host__ __device__ constexpr size_t pass_smem_x()
{
    return N % 16 == 0 ? pass_smem_strided<N, T>() : 2 * sizeof(float2) * N * PAIRS + 2 * sizeof(float2) * N;
}

// Tensor memory as a per-thread store: K consecutive columns of the thread's lane.
// The instructions are .aligned, all 32 lanes at once, while the loops around them
// branch by lane (a ragged tile's missing lines, PML rows): each helper brings the
// warp together first.
template <int K>
__device__ __forceinline__ void tmem_st(uint32_t addr, const float* v)
{
    static_assert(K == 4 || K == 8, "");
    __syncwarp();
    if constexpr (K == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr),
                     "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[0]), "f"(v[1]),
                     "f"(v[2]), "f"(v[3])
                     : "memory");
}
__device__ __forceinline__ void tmem_st_wait()
{
    __syncwarp();
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
template <int K>
__device__ __forceinline__ void tmem_ld(uint32_t addr, float* v)
{
    static_assert(K == 4 || K == 8, "");
    __syncwarp();
    if constexpr (K == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                     "tcgen05.wait::ld.sync.aligned;"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                     : "r"(addr)
                     : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\ntcgen05.wait::ld.sync.aligned;"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "r"(addr)
                     : "memory");
}
// warp 0 takes the CTA's columns (it waits while other CTAs hold them: they
// give them back without waiting for this one) and publishes the address
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, unsigned columns)
{
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(slot)),
                 "r"(columns)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, unsigned columns)
{
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(columns) : "memory");
}

// Programmatic dependent launch (a pass launched with PDL while the previous
// pass of the same half-step drains): let the next pass launch once every CTA
// of this one has started, and wait for the previous pass to complete (and its
// writes to be visible) before touching what it writes.  Both are no-ops for a
// plain launch.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Start of a pass.  pdl 2: wait for the previous kernel first, and only then
// let dependents launch, so a dependent that reads early never overtakes a
// kernel this one still waits for.  pdl 1: this pass's early reads are final
// already (it launched after the previous pass had passed its own wait), so
// dependents may launch at once; the epilogue waits (pdl_wait) before adding.
// pdl 0: a plain launch, dependents launch when it completes.
__device__ __forceinline__ void pdl_begin(int pdl)
{
    if (pdl == 2) pdl_wait();
    if (pdl != 0) pdl_launch_dependents();
}

// Launch of a pass kernel, with the programmatic-stream-serialization
// attribute when p.pdl is set (the kernel then waits as p.pdl says).
template <class K, class... Args>
inline cudaError_t launch_pass_kernel(K kernel, dim3 grid, int threads, size_t smem, cudaStream_t st,
                                      const PassParams& p, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p, args...);
}

// CTAs of a persistent launch over `units` tiles: what the device holds at
// once (by shared memory, registers and threads), or fewer so that all of them
// take the same number of tiles
template <class K>
inline cudaError_t persistent_grid(K kernel, int threads, size_t smem, int units, int* grid)
{
    int dev = 0, sms = 0, sm_smem = 0, sm_regs = 0, sm_threads = 0, reserved = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_threads, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    const int warps = (threads + 31) / 32;
    const int per_warp = (fa.numRegs + 7) / 8 * 8 * 32;  // registers are given out in eights per thread
    int per = std::min(sm_threads / (32 * warps), sm_regs / (per_warp * warps));
    per = std::min(per, (int)(sm_smem / (smem + fa.sharedSizeBytes + reserved)));
    const int most = sms * std::max(1, per);
    const int rounds = (units + most - 1) / most;
    *grid = (units + rounds - 1) / rounds;
    return cudaSuccess;
}

// Fused point sources and receivers of this CTA (PassParams::sp_mode): once
// the CTA's own field updates are done (a CTA barrier makes its threads'
// reductions visible to the CTA; the reads go through L2), thread 0 adds the
// sources in their order, and after a second barrier every receiver is
// recorded by a thread of its own -- the arithmetic of the separate injection
// and recording kernels (inject_kernel, record_kernel).  job and tile: those of
// the tile just updated (StridedTile::job, ::list): the velocity z pass's job c updates
// v_c, the stress y pass's job 1 sxy, the stress z pass's job 0 sxx syy szz, job 1
// sxz, job 2 syz.
__device__ __forceinline__ void special_phase(const PassParams& p, const PassJob& J, int job, int tile)
{
    const int b0 = p.sp_off[tile], b1 = p.sp_off[tile + 1];
    if (b0 == b1) return;  // the same for every thread of the CTA
    const int n = *p.step_now - 1;
    __syncthreads();
    if (p.sp[b0].kind != SP_RECEIVER) {  // sources come first in the list
        if (threadIdx.x == 0) {
            if (p.pdl == 1) pdl_wait();  // (done already if this thread had cells to update)
            for (int e = b0; e < b1; ++e) {
                if (!ES_INB(p, e, p.ext_sp)) break;
                const SpecialCell c = p.sp[e];
                if (c.kind == SP_RECEIVER) break;
                const SourceDev& s = p.src[c.idx];
                if (n >= s.nw) continue;
                const float w = s.w[n];
                auto add = [&](float* t, float m) {
                    if (m != 0.f && ES_INB(p, c.q, p.ext_f)) *t = __fmaf_rn(m, w, __ldcg(t));
                };
                if (p.sp_mode == SP_VEL_Z) {
                    if (c.kind == SP_FORCE) add(J.tgt[0] + c.q, s.m[job]);
                } else if (c.kind == SP_MOMENT) {
                    if (p.sp_mode == SP_STR_Y) {
                        if (job == 1) add(J.tgt[0] + c.q, s.m[3]);
                    } else if (job == 0) {
                        add(J.tgt[0] + c.q, s.m[0]);
                        add(J.tgt[1] + c.q, s.m[1]);
                        add(J.tgt[2] + c.q, s.m[2]);
                    } else {
                        add(J.tgt[0] + c.q, s.m[job == 1 ? 4 : 5]);
                    }
                }
            }
        }
        __syncthreads();
    }
    if (p.sp_mode == SP_STR_Y || (p.sp_mode == SP_STR_Z && job != 0)) return;
    if (p.pdl == 1) pdl_wait();
    for (int e = b0 + threadIdx.x; e < b1; e += blockDim.x) {
        if (!ES_INB(p, e, p.ext_sp)) break;
        const SpecialCell c = p.sp[e];
        if (c.kind != SP_RECEIVER) continue;
        const size_t row0 = ((size_t)(n - p.rec_start) * p.nsim + c.sim) * 4 * p.n_rcv;
        if (!ES_INB(p, c.q, p.ext_f) || !ES_INB(p, row0 + 4 * (size_t)p.n_rcv - 1, p.ext_rec)) continue;
        float* row = p.rec + row0;
        if (p.sp_mode == SP_VEL_Z) {
            row[(size_t)(job + 1) * p.n_rcv + c.idx] = __ldcg(J.tgt[0] + c.q);
        } else {
            const float s = __fadd_rn(__fadd_rn(__ldcg(J.tgt[0] + c.q), __ldcg(J.tgt[1] + c.q)),
                                      __ldcg(J.tgt[2] + c.q));
            row[c.idx] = __fdiv_rn(-s, 3.f);  // Eq. (3)
        }
    }
}

// warm L2 with a 128-byte line the epilogue will read (no registers held)
__device__ __forceinline__ void prefetch_l2(const void* p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// twiddles and the multiplier of this job's direction into shared memory
template <int N>
__device__ __forceinline__ void load_tables(const PassParams& p, const PassJob& J, float2* s_tw, float2* s_h, int tid,
                                            int nthreads)
{
    const float2* h = J.sign > 0 ? p.hp : p.hm;
    for (int i = tid; i < N; i += nthreads) {
        s_tw[i] = __ldg(p.tw + i);
        s_h[i] = __ldg(h + i);
    }
}

// Near part of the rows RA j .. RA j + RA - 1 of pair c: the NEAR_TAPS taps in
// order from the first offset, the window of rows sliding through registers,
// wrapped along the axis.  row(e) reads source row e of this pair, put(q, s)
// takes the result of row RA j + q.
template <int N, int RA, class Row, class Put>
__device__ __forceinline__ void near_part(const PassJob& J, int j, Row row, Put put)
{
    const int ofs = near_ofs(J.sign);
    float2 g[NEAR_TAPS];
#pragma unroll
    for (int t = 0; t < NEAR_TAPS; ++t) g[t] = rep2(J.g[t]);
    float2 w[RA + NEAR_TAPS - 1];
#pragma unroll
    for (int k = 0; k < RA + NEAR_TAPS - 1; ++k) {
        int e = RA * j + ofs + k;
        if (k < 5) e = e < 0 ? e + N : e;             // the first rows of the axis look back over its end,
        if (k >= RA + 4) e = e >= N ? e - N : e;      // the last ones past it (ofs is -4 or -5)
        w[k] = row(e);
        if (k >= NEAR_TAPS - 1) {
            const int q = k - (NEAR_TAPS - 1);
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int t = 0; t < NEAR_TAPS; ++t) s = fma2(g[t], w[q + t], s);
            put(q, s);
        }
    }
}

// A tile of a y or z pass: 32 consecutive x at one z (y pass) or one y (z
// pass) of one simulation, and the job done on it.
struct StridedTile {
    int job, list;   // list: index of the tile in the special-cell lists
    int x0, outer;
    size_t base;     // linear index of its first cell
    size_t off, soff;
};
template <int PR = PAIRS>
__device__ __forceinline__ StridedTile strided_tile(const PassParams& p, int w, int ntiles)
{
    StridedTile t;
    t.job = 0;
    while (w >= ntiles) {  // at most njobs - 1 times
        w -= ntiles;
        ++t.job;
    }
    t.list = w;
    // simulations run fastest: the CTAs of one tile are adjacent and read that
    // tile's material rows through L2
    int sim = 0;
    if (p.nsim > 1) {
        sim = w % p.nsim;
        w /= p.nsim;
    }
    const int ntx = (p.nx + 2 * PR - 1) / (2 * PR);
    t.outer = w / ntx;
    t.x0 = (w - t.outer * ntx) * 2 * PR;
    t.base = (size_t)t.x0 + (size_t)p.nx * (p.axis == 1 ? (size_t)p.ny * t.outer : (size_t)t.outer);
    t.off = (size_t)sim * p.fstride;
    t.soff = (size_t)sim * p.sstride;
    return t;
}

// the tile's source into shared rows, W floats per asynchronous copy, zeros
// past the last column
template <int NT, int W, int PR = PAIRS>
__device__ __forceinline__ void stage_strided(const PassParams& p, const StridedTile& t, float2* buf, unsigned est,
                                              int n)
{
    constexpr int CH = W == 1 ? PR : 2 * PR / W;  // threads per row
    static_assert(NT % CH == 0, "a thread keeps its columns");
    const float* src = p.job[t.job].src + t.off + t.base;
    const int e0 = threadIdx.x / CH, k = threadIdx.x % CH;
    // floats of a row this thread copies: W from x0 + W k on; W = 1: x0 + k and x0 + PR + k, the
    // two pencils of pair k
    const int x = W * k;
    unsigned o = (unsigned)e0 * est + x;
    float* d = reinterpret_cast<float*>(buf + e0 * PR) + (W == 1 ? 2 * k : x);
#pragma unroll 4
    for (int e = e0; e < n; e += NT / CH, o += NT / CH * est, d += NT / CH * 2 * PR) {
#pragma unroll
        for (int f = 0; f < (W == 1 ? 2 : 1); ++f) {
            const bool ok = t.x0 + x + f * PR < p.nx && ES_INB(p, t.off + t.base + o + f * PR + W - 1, p.ext_f);
            cp_async<4 * W>(d + f, ok ? src + o + f * PR : src, ok);
        }
    }
}

// Epilogue of a tile of a y or z pass: each thread takes RN consecutive
// positions of its pair, EB at a time with the next batch's coefficients in
// flight; the far parts come from the shared rows, the near parts from tensor
// memory (TM) or their shared rows.  Addresses are a tile's base plus a 32-bit
// offset.  FULL: the threads' positions are exactly the axis (else they may pass
// its end).
//
// The PML slab rows (the first L and the last L + 1 positions) would all fall to
// the first and the last warps, which would keep the others waiting while they
// fetch the old splits: there the derivative goes back into the shared row, and
// afterwards the CTA takes the slab's (row, pair) items evenly (run_slab).
template <int RN, int V, bool TM, bool FULL = true, int PR = PAIRS>
struct StridedEpilogue {
    static constexpr int EB = epi_batch<RN>();
    const PassParams& p;
    const PassJob& J;
    const StridedTile& t;
    const unsigned est;
    float2* const rows;   // the far parts (source tile's rows)
    const float2* const near;
    const uint32_t tm;
    const int c, pos0;
    const bool valid, two;
    const float *co0, *co1;
    unsigned o;
    float2 c0[EB], c1[EB];

    __device__ __forceinline__ StridedEpilogue(const PassParams& p_, const PassJob& J_, const StridedTile& t_,
                                               unsigned est_, float2* buf, const float2* nearp, uint32_t tm_)
        : p(p_), J(J_), t(t_), est(est_), rows(buf), near(nearp), tm(tm_), c((int)threadIdx.x % PR),
          pos0(RN * ((int)threadIdx.x / PR)), valid(t_.x0 + V * c < p_.nx), two(V == 2 || t_.x0 + PR + c < p_.nx)
    {
        co0 = J.coef[0] + t.base;
        co1 = J.coef[1] + t.base;
        o = (unsigned)pos0 * est + V * c;
    }
    // whether this thread updates its k-th position
    __device__ __forceinline__ bool in(int k) const { return valid && (FULL || pos0 + k < p.n); }
    __device__ __forceinline__ void coefs(int oc0, unsigned oc, bool normal)
    {
#pragma unroll
        for (int e = 0; e < EB; ++e) {
            const unsigned oe = oc + e * est;
            if (!in(oc0 + e) || !ES_INB(p, t.base + oe + last(), p.ext_c)) continue;
            c0[e] = ldg_pair<V, PR>(co0 + oe, two);
            if (normal) c1[e] = ldg_pair<V, PR>(co1 + oe, two);
        }
    }
    __device__ __forceinline__ void first_coefs()
    {
        if (J.kind != JOB_STORE) coefs(0, o, J.kind == JOB_NORMAL);
    }
    // offset of the pair's last cell (index checks)
    __device__ __forceinline__ int last() const { return V == 2 ? 1 : (two ? PR : 0); }
    // SLAB: slab rows may be among this warp's positions
    template <int KIND, bool SLAB>
    __device__ __forceinline__ void run()
    {
        constexpr int NT = KIND == JOB_NORMAL ? 3 : 1;
        float* tgt[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) tgt[k] = J.tgt[k] + t.off + t.base;
        const float dt = p.dt;
#pragma unroll 1
        for (int k0 = 0; k0 < RN; k0 += EB) {
            float s[2 * EB];
            if constexpr (TM) tmem_ld<2 * EB>(tm + (uint32_t)(2 * k0), s);
            float2 d0[EB], d1[EB];
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                d0[e] = c0[e];
                d1[e] = c1[e];
            }
            if (KIND != JOB_STORE && k0 + EB < RN) coefs(k0 + EB, o + EB * est, KIND == JOB_NORMAL);
#pragma unroll
            for (int e = 0; e < EB; ++e, o += est) {
                const int pos = pos0 + k0 + e;
                float2* const row = rows + pos * PR + c;
                const float2 f = *row;
                // (past the axis's end the near parts have no row)
                const float2 n = TM ? make_float2(s[2 * e], s[2 * e + 1])
                                    : (FULL || pos < p.n ? near[pos * PR + c] : make_float2(0.f, 0.f));
                const float2 d = make_float2(__fadd_rn(f.x, n.x), __fsub_rn(n.y, f.y));  // far (conj) + near
                const bool ok = in(k0 + e) && ES_INB(p, t.off + t.base + o + last(), p.ext_f);
                if (KIND == JOB_STORE) {
                    if (ok) st_pair<V, PR>(tgt[0] + o, d, two);
                    continue;
                }
#if ES_BOUNDS
                if (!ok || !ES_INB(p, t.base + o + last(), p.ext_c)) continue;
#endif
                if (SLAB && in_slab(pos, p.n, p.L)) {
                    if (FULL || pos < p.n) *row = d;
                    continue;
                }
#pragma unroll
                for (int k = 0; k < NT; ++k) {
                    const bool diag = k == J.diag;
                    const float cx = KIND == JOB_NORMAL ? normal_coef(d0[e].x, d1[e].x, diag) : d0[e].x;
                    const float cy = KIND == JOB_NORMAL ? normal_coef(d0[e].y, d1[e].y, diag) : d0[e].y;
                    const float2 inc = make_float2(increment(dt, cx, d.x), increment(dt, cy, d.y));
                    if (ok) red_pair<V, PR>(tgt[k] + o, inc, two);
                }
            }
        }
    }
    // the slab rows, (row, pair) items dealt over the CTA's NTHR threads
    template <int KIND, int NTHR>
    __device__ __forceinline__ void run_slab()
    {
        constexpr int NT = KIND == JOB_NORMAL ? 3 : 1;
        const int S = 2 * p.L + 1;
        const float* prof = J.stag ? p.ps : p.pc;
        // slab rows have the field's stride along the axis
        const size_t s0 = t.soff + t.x0 + (p.axis == 1 ? (size_t)p.nx * S * t.outer : (size_t)p.nx * t.outer);
        if (!valid) return;
#pragma unroll 1
        for (int sp = threadIdx.x / PR; sp < S; sp += NTHR / PR) {
            const int pos = sp < p.L ? sp : sp - p.L + p.n - 1 - p.L;
            const unsigned q = (unsigned)pos * est + V * c, so = (unsigned)sp * est + V * c;
            if (!ES_INB(p, t.off + t.base + q + last(), p.ext_f) ||
                !ES_INB(p, t.base + q + last(), p.ext_c) || !ES_INB(p, s0 + so + last(), p.ext_s))
                continue;
            const float2 d = rows[pos * PR + c];
            const float2 k0 = ldg_pair<V, PR>(co0 + q, two);
            const float2 k1 = KIND == JOB_NORMAL ? ldg_pair<V, PR>(co1 + q, two) : k0;
            const float P = __ldg(prof + pos);
            float2 sv[NT];
#pragma unroll
            for (int k = 0; k < NT; ++k) sv[k] = ld_pair<V, PR>(J.slab[k] + s0 + so, two);
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                const bool diag = k == J.diag;
                const float cx = KIND == JOB_NORMAL ? normal_coef(k0.x, k1.x, diag) : k0.x;
                const float cy = KIND == JOB_NORMAL ? normal_coef(k0.y, k1.y, diag) : k0.y;
                float2 inc = make_float2(increment(p.dt, cx, d.x), increment(p.dt, cy, d.y));
                // split-field update s <- P (P s + inc); the total takes the split's change
                const float2 sn = make_float2(__fmul_rn(P, __fmaf_rn(P, sv[k].x, inc.x)),
                                              __fmul_rn(P, __fmaf_rn(P, sv[k].y, inc.y)));
                st_pair<V, PR>(J.slab[k] + s0 + so, sn, two);
                inc = make_float2(__fsub_rn(sn.x, sv[k].x), __fsub_rn(sn.y, sv[k].y));
                red_pair<V, PR>(J.tgt[k] + t.off + t.base + q, inc, two);
            }
        }
    }
};

// y and z passes, persistent: CTA b takes tiles b, b + gridDim.x, ... of
// njobs x ntiles (job slowest), and while it works on one, the next one's source
// arrives in the other half of its shared memory.  V: floats per access of the
// epilogue (2: nx even; 1: nx odd).
template <int RA, int RB, int RC, int T, int V>
__global__ void __launch_bounds__(pass_threads<T>(), pass_min_blocks<RA, RB, RC, T>())
pass_strided(const __grid_constant__ PassParams p, int ntiles)
{
    using C = CoreOf<RA, RB, RC, T>;
    constexpr int N = C::N, RN = N / T, NT = T * PAIRS;
    constexpr bool TM = near_in_tmem<N, T>();
    constexpr int EB = epi_batch<RN>();
    extern __shared__ __align__(16) float2 smem[];
    __shared__ uint32_t tmem_slot;
    float2* nearp = smem + 2 * N * PAIRS;  // near parts (not TM)
    float2* s_tw = nearp + (TM ? 0 : N * PAIRS);
    float2* s_hp = s_tw + N;
    float2* s_hm = s_hp + N;
    const int tid = threadIdx.x;
    const int c = tid % PAIRS, j = tid / PAIRS;
    uint32_t tm = 0;
    // the columns are taken before dependents may launch: a dependent kernel's
    // CTAs, which may hold columns while they wait for this kernel, then never
    // keep them from it
    if (TM) {
        if (tid < 32) tmem_alloc(&tmem_slot, tmem_columns<N, T>());
        __syncthreads();
        tm = tmem_slot + ((uint32_t)(tid / 32 % 4) << 21) + (uint32_t)(tid / 128 * 2 * RN);
    }
    pdl_begin(p.pdl);
    // stride along the axis; offsets within a tile fit 32 bits (an axis has at most 512 cells)
    const unsigned est = p.axis == 1 ? (unsigned)p.nx : (unsigned)p.nx * p.ny;
    const int total = ntiles * p.njobs;
    auto stage = [&](const StridedTile& t, float2* buf) {
        if (V == 1) stage_strided<NT, 1>(p, t, buf, est, N);
        else if (p.nx % 4 == 0) stage_strided<NT, 4>(p, t, buf, est, N);
        else stage_strided<NT, 2>(p, t, buf, est, N);
    };
    stage(strided_tile(p, blockIdx.x, ntiles), smem);
    for (int i = tid; i < N; i += NT) {
        s_tw[i] = __ldg(p.tw + i);
        s_hp[i] = __ldg(p.hp + i);
        s_hm[i] = __ldg(p.hm + i);
    }
    bool waited = p.pdl != 1;
    int half = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x, half ^= 1) {
        const PassJob& J = p.job[w / ntiles];
        float2* buf = smem + half * N * PAIRS;
        cp_async_commit_wait_all();
        __syncthreads();  // the tile is there; the other half is no longer read
        if (w + (int)gridDim.x < total)
            stage(strided_tile(p, w + gridDim.x, ntiles), smem + (half ^ 1) * N * PAIRS);
        // coefficient and PML slab rows of this tile (128 bytes each) into L2 for the epilogue
        if (J.coef[0]) {
            const StridedTile t = strided_tile(p, w, ntiles);
            for (int i = tid; i < N; i += NT) {
                const unsigned o = (unsigned)i * est;
                if (ES_INB(p, t.base + o, p.ext_c)) {
                    prefetch_l2(J.coef[0] + t.base + o);
                    if (J.coef[1]) prefetch_l2(J.coef[1] + t.base + o);
                }
            }
            const int S = p.L > 0 ? 2 * p.L + 1 : 0;
            const size_t s0 = t.soff + t.x0 + (p.axis == 1 ? (size_t)p.nx * S * t.outer : (size_t)p.nx * t.outer);
            for (int i = tid; i < S; i += NT) {
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
        if constexpr (TM) {
            float v[2 * EB];
            near_part<N, RN>(
                J, j, [&](int e) { return buf[e * PAIRS + c]; },
                [&](int q, float2 s) {
                    v[2 * (q % EB)] = s.x;
                    v[2 * (q % EB) + 1] = s.y;
                    if (q % EB == EB - 1) tmem_st<2 * EB>(tm + (uint32_t)(2 * (q - EB + 1)), v);
                });
        } else {
            near_part<N, RN>(
                J, j, [&](int e) { return buf[e * PAIRS + c]; },
                [&](int q, float2 s) { nearp[(RN * j + q) * PAIRS + c] = s; });
        }
        {
            float2 a[C::MA][RA];
            C::stageA(a, j, [&](int e) { return buf[e * PAIRS + c]; });
            __syncthreads();  // the source rows have been read
            C::stageA_store(a, buf, j, c);
            __syncthreads();
            C::middle(buf, s_tw, J.sign > 0 ? s_hp : s_hm, j, c);
            __syncthreads();
            C::stageA_inv(buf, s_tw, a, j, c);
            __syncthreads();  // the FFT's rows have been read
            C::results(a, j, [&](int e, float2 v) { buf[e * PAIRS + c] = v; });
        }
        if (TM) tmem_st_wait();
        // epilogue of the positions RN j .. RN j + RN - 1 of the thread's pair: one variant per kind
        // of job and, for whole warps, with or without PML slab rows among their positions
        const StridedTile t = strided_tile(p, w, ntiles);
        StridedEpilogue<RN, V, TM> ep(p, J, t, est, buf, nearp, tm);
        const int r0 = RN * (tid / 32 * (32 / PAIRS)), r1 = r0 + RN * (32 / PAIRS);  // rows of this warp
        const bool slab = p.L > 0 && (r0 < p.L || r1 > p.n - 1 - p.L);
        ep.first_coefs();
        __syncthreads();  // the far parts are there
        if (!waited) {
            pdl_wait();  // the previous pass's updates of the targets come first
            waited = true;
        }
        if (J.kind == JOB_STORE) ep.template run<JOB_STORE, false>();
        else if (J.kind == JOB_SINGLE && !slab) ep.template run<JOB_SINGLE, false>();
        else if (J.kind == JOB_SINGLE) ep.template run<JOB_SINGLE, true>();
        else if (!slab) ep.template run<JOB_NORMAL, false>();
        else ep.template run<JOB_NORMAL, true>();
        if (p.L > 0 && J.kind != JOB_STORE) {
            __syncthreads();
            if (J.kind == JOB_SINGLE) ep.template run_slab<JOB_SINGLE, NT>();
            else ep.template run_slab<JOB_NORMAL, NT>();
        }
        if (p.sp_mode != SP_NONE) special_phase(p, J, t.job, t.list);
    }
    if (TM) {
        __syncthreads();
        if (tid < 32) tmem_free(tmem_slot, tmem_columns<N, T>());
    }
}

// The same passes with one tile per CTA (blockIdx.x) and job (blockIdx.y), for the shortest lengths and
// the odd ones: the source goes straight into registers and comes again, from L2, for the stencil once
// the FFT is done with the one shared tile, so a CTA takes a third of the shared memory and more of them
// hide each other's chain of loads and stages.  A thread keeps the elements its first stage reads, j + q
// N / RA, to the end.  Which lengths: one_tile(), pass_strided.cuh.
constexpr int HALO = 5;  // rows of wrap-around copies on each side of that tile
static_assert(-near_ofs(-1) <= HALO && near_ofs(+1) + NEAR_TAPS - 1 <= HALO, "near taps reach beyond the halo");
template <int RA, int RB, int RC>
__host__ __device__ constexpr int once_threads() { return RB * RC * PAIRS; }
// (more threads than the register file holds at 64 each, but for the butterflies that need those: 75 = 5 x
// 15 with four and five CTAs per SM 70.6 and 65.4 ps per cell, 64 = 16 x 4 with 16 and 18 50.9 and 59.5)
template <int RA, int RB, int RC>
__host__ __device__ constexpr int once_blocks() { return (RA <= 12 ? 1200 : 1024) / once_threads<RA, RB, RC>(); }
template <int RA, int RB, int RC>
__host__ __device__ constexpr size_t once_smem()
{
    return sizeof(float2) * ((size_t)(RA * RB * RC + 2 * HALO) * PAIRS + 2 * (size_t)RA * RB * RC);
}

// Update of one pair of cells: offsets of its first cell in a field (f), a coefficient array (cf) and a slab
// array (s: of slab coordinate 0, est per coordinate), position pos along the axis.
template <int V>
__device__ __forceinline__ void update_pair(const PassParams& p, const PassJob& J, size_t f, size_t cf, size_t s, unsigned est,
                                            int pos, float2 d, bool two)
{
    const int last = V == 2 ? 1 : (two ? PAIRS : 0);
    if (!ES_INB(p, f + last, p.ext_f)) return;
    if (J.kind == JOB_STORE) {
        st_pair<V, PAIRS>(J.tgt[0] + f, d, two);
        return;
    }
    if (!ES_INB(p, cf + last, p.ext_c)) return;
    const bool slab = in_slab(pos, p.n, p.L);
    float P = 1.f;
    if (slab) {
        s += (size_t)((unsigned)slab_pos(pos, p.n, p.L, p.S) * est);
        if (!ES_INB(p, s + last, p.ext_s)) return;
        P = __ldg((J.stag ? p.ps : p.pc) + pos);
    }
    auto add = [&](int k, float2 c) {
        float2 inc = make_float2(increment(p.dt, c.x, d.x), increment(p.dt, c.y, d.y));
        if (slab) {  // s <- P (P s + inc); the total takes the split's change
            const float2 sv = ld_pair<V, PAIRS>(J.slab[k] + s, two);
            const float2 sn = make_float2(__fmul_rn(P, __fmaf_rn(P, sv.x, inc.x)), __fmul_rn(P, __fmaf_rn(P, sv.y, inc.y)));
            st_pair<V, PAIRS>(J.slab[k] + s, sn, two);
            inc = make_float2(__fsub_rn(sn.x, sv.x), __fsub_rn(sn.y, sv.y));
        }
        red_pair<V, PAIRS>(J.tgt[k] + f, inc, two);
    };
    const float2 c0 = ldg_pair<V, PAIRS>(J.coef[0] + cf, two);
    if (J.kind == JOB_SINGLE) {
        add(0, c0);
    } else {
        const float2 c1 = ldg_pair<V, PAIRS>(J.coef[1] + cf, two);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            add(k, make_float2(normal_coef(c0.x, c1.x, k == J.diag), normal_coef(c0.y, c1.y, k == J.diag)));
    }
}

template <int RA, int RB, int RC, int V>
__global__ void __launch_bounds__(once_threads<RA, RB, RC>(), once_blocks<RA, RB, RC>())
pass_strided_once(const __grid_constant__ PassParams p, int ntiles)
{
    constexpr int T = RB * RC, NT = T * PAIRS;
    using C = CoreOf<RA, RB, RC, T>;
    constexpr int N = C::N, BA = C::BA;
    static_assert(C::MA == 1, "a thread's elements are j + q BA");
    extern __shared__ __align__(16) float2 smem[];
    float2* buf = smem;  // FFT rows 0 .. N-1; then the source tile at rows HALO + pos (wrapped)
    float2* s_tw = buf + (N + 2 * HALO) * PAIRS;
    float2* s_h = s_tw + N;
    const int tid = threadIdx.x;
    const int c = tid % PAIRS, j = tid / PAIRS;
    const PassJob& J = p.job[blockIdx.y];
    pdl_begin(p.pdl);
    const unsigned est = p.axis == 1 ? (unsigned)p.nx : (unsigned)p.nx * p.ny, step = BA * est;
    const StridedTile t = strided_tile(p, blockIdx.x, ntiles);
    const bool valid = t.x0 + V * c < p.nx, two = V == 2 || t.x0 + PAIRS + c < p.nx;
    const int last = V == 2 ? 1 : (two ? PAIRS : 0);
    const size_t f0 = t.off + t.base + V * c;
    const float* src = J.src + f0;
    float2 a[1][RA];
#pragma unroll
    for (int q = 0; q < RA; ++q)
        a[0][q] = valid && ES_INB(p, f0 + (j + q * BA) * est + last, p.ext_f)
                      ? ldg_pair<V, PAIRS>(src + (j + q * BA) * est, two)
                      : make_float2(0.f, 0.f);
    // coefficient rows of this tile (128 bytes each) into L2 for the epilogue
    if (J.coef[0])
        for (int i = tid; i < N; i += NT) {
            const unsigned o = (unsigned)i * est;
            if (ES_INB(p, t.base + o, p.ext_c)) {
                prefetch_l2(J.coef[0] + t.base + o);
                if (J.coef[1]) prefetch_l2(J.coef[1] + t.base + o);
            }
        }
    load_tables<N>(p, J, s_tw, s_h, tid, NT);
    Dft<RA>::run(a[0]);
    C::stageA_store(a, buf, j, c);
    __syncthreads();
    C::middle(buf, s_tw, s_h, j, c);
    __syncthreads();
    C::stageA_inv(buf, s_tw, a, j, c);
    __syncthreads();  // the FFT's rows have been read
    auto copy = [&](float2* d, unsigned o) {
        if (!ES_INB(p, f0 + o + last, p.ext_f)) return;
        if constexpr (V == 2) {
            cp_async<8>(d, src + o, true);
        } else {
            cp_async<4>(&d->x, src + o, true);
            cp_async<4>(&d->y, two ? src + o + PAIRS : src, two);
        }
    };
    if (valid) {
        unsigned o = (unsigned)j * est;
        float2* d = buf + (j + HALO) * PAIRS + c;
#pragma unroll 1
        for (int q = 0; q < RA; ++q, o += step, d += BA * PAIRS) copy(d, o);
        for (int h = j; h < 2 * HALO; h += T) {
            const int pos = h < HALO ? N - HALO + h : h - HALO;
            copy(buf + (h < HALO ? h : N + h) * PAIRS + c, (unsigned)pos * est);
        }
    }
    cp_async_commit_wait_all();
    __syncthreads();
    if (valid) {
        const float2* w = buf + (j + HALO + near_ofs(J.sign)) * PAIRS + c;
#pragma unroll
        for (int q = 0; q < RA; ++q) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NEAR_TAPS; ++k) s = fma2(rep2(J.g[k]), w[(q * BA + k) * PAIRS], s);
            a[0][q] = make_float2(__fadd_rn(a[0][q].x, s.x), __fsub_rn(s.y, a[0][q].y));  // far (conj) + near
        }
        if (p.pdl == 1) pdl_wait();  // the previous pass's updates of the targets come first
        const size_t s0 = t.soff + t.x0 + V * c + (p.axis == 1 ? (size_t)p.nx * p.S * t.outer : (size_t)p.nx * t.outer);
#pragma unroll
        for (int q = 0; q < RA; ++q)
            update_pair<V>(p, J, f0 + (j + q * BA) * est, t.base + V * c + (j + q * BA) * est, s0, est, j + q * BA, a[0][q], two);
    }
    if (p.sp_mode != SP_NONE) special_phase(p, J, blockIdx.y, t.list);
}

// x pass: cell (position x, line r of the tile) of a turned-around tile is
// float x_at(x, r): row x, the line exchanged within the row (whole pairs) so
// that the turning accesses of a warp, x_chunks 4-cell chunks of 32 / x_chunks
// lines (lengths that are a multiple of 16) or 8 cells of 4 lines (others), hit
// 32 banks.
template <int N>
__host__ __device__ constexpr int x_chunks()
{
    return N % 32 == 0 ? 8 : 4;
}
template <int N>
__device__ __forceinline__ int x_swz(int x)
{
    return N % 32 == 0 ? ((x >> 2) & 7) << 1 : (N % 16 == 0 ? ((x >> 2) & 3) << 2 : (x & 7) << 1);
}
template <int N>
__device__ __forceinline__ int x_at(int x, int r)
{
    return x * 2 * PAIRS + (r ^ (x_swz<N>(x) << 1));
}

// An item of the x pass (lengths that are a multiple of 16): four consecutive
// cells xx .. xx + 3 of line r of the tile
template <int N>
__device__ __forceinline__ void x_item(int it, int* r, int* xx)
{
    constexpr int CL = x_chunks<N>();
    const int lo = it % CL;
    *r = (it / CL) % (2 * PAIRS);
    *xx = 4 * (it / (CL * 2 * PAIRS) * CL + lo);
}

// The cells of an x-pass tile in memory order that are updated four at a time: nq chunks of four from the
// h-th of its nf cells on, where the targets reach a 16-byte boundary (a simulation of an odd cell count
// starts off one); on: from the first cell on, and the coefficients are on one too.  Tiles off a boundary
// went cell by cell, a chain of coefficient, split and target for each: us a velocity and a stress x pass
// (one GB300), five simulations of 14 x 75 x 75 28.2 and 33.4 -> 18.5 and 20.3, two of 75^3 36.2 and 40.9 -> 25.7
// and 26.6; batches of 66 and 127 cells as convolutions 32.1 and 36.7 -> 25.6 and 27.8, 26.7 and 31.0 -> 19.6 and
// 21.6 ps per cell.  The loops stay apart: one for both cost aligned 125-cell tiles 8 % in registers.
struct XQuads {
    int h, nq;
    bool on;
};
__device__ __forceinline__ XQuads x_quads(const PassJob& J, size_t off, size_t q0, int nf)
{
    auto mis = [](const float* q) { return (int)((uintptr_t)q >> 2) & 3; };  // floats past the last boundary
    const int m = mis(J.tgt[0] + off + q0);
    XQuads x = {min((4 - m) & 3, nf), 0, m == 0};
    bool same = true;
    if (J.kind == JOB_NORMAL) {
        same = mis(J.tgt[1] + off + q0) == m && mis(J.tgt[2] + off + q0) == m;
        x.on = x.on && mis(J.coef[1] + q0) == 0;
    }
    if (J.kind != JOB_STORE) x.on = x.on && mis(J.coef[0] + q0) == 0;
    if (same) x.nq = (nf - x.h) / 4;
    else x.h = 0;
    return x;
}

// Update of those chunks, the next one's coefficients in flight (ON: XQuads::on; else four loads each).  A
// chunk may span two lines, so every cell takes its own x and line for the PML split.
template <int NT, int KIND, bool ON, class LineOf>
__device__ __forceinline__ void x_quads_flat(const PassParams& p, const PassJob& J, const float* bf, size_t q0, int line0,
                                             const XQuads& xq, int n, size_t off, size_t soff, LineOf line_of)
{
    constexpr int TG = KIND == JOB_NORMAL ? 3 : 1;
    const int nq = xq.nq, h = ON ? 0 : xq.h;
    q0 += h;
    bf += h;
    const float *co0 = J.coef[0] + q0, *co1 = J.coef[1] + q0;
    const float* prof = J.stag ? p.ps : p.pc;
    float* tgt[TG];
#pragma unroll
    for (int k = 0; k < TG; ++k) tgt[k] = J.tgt[k] + off + q0;
    float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0;
    auto four = [](const float* q) {
        if constexpr (ON) return __ldg(reinterpret_cast<const float4*>(q));
        else return make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), __ldg(q + 3));
    };
    auto coefs = [&](int i) {
        if (KIND == JOB_STORE || i >= nq || !ES_INB(p, q0 + 4 * i + 3, p.ext_c)) return;
        c0 = four(co0 + 4 * i);
        if (KIND == JOB_NORMAL) c1 = four(co1 + 4 * i);
    };
    coefs(threadIdx.x);
#pragma unroll 1
    for (int i = threadIdx.x; i < nq; i += NT) {
        const float4 a4 = c0, b4 = c1;
        const float4 d4 = ON ? reinterpret_cast<const float4*>(bf)[i]
                             : make_float4(bf[4 * i], bf[4 * i + 1], bf[4 * i + 2], bf[4 * i + 3]);
        coefs(i + NT);
        if (!ES_INB(p, off + q0 + 4 * i + 3, p.ext_f)) continue;
        if (KIND == JOB_STORE) {
            reinterpret_cast<float4*>(tgt[0])[i] = d4;
            continue;
        }
        const float d[4] = {d4.x, d4.y, d4.z, d4.w}, a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
        // the cells' split parts, all on their way before the first is used
        size_t si[4];
        float P[4], old[TG][4];
        unsigned slab = 0;
        if (p.L > 0) {
            const int f = h + 4 * i, r = line_of(f), x = f - r * n;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int xe = x + e < n ? x + e : x + e - n, re = x + e < n ? r : r + 1;
                if (!in_slab(xe, n, p.L)) continue;
                si[e] = soff + (size_t)p.S * (line0 + re) + slab_pos(xe, n, p.L, p.S);
                if (!ES_INB(p, si[e], p.ext_s)) continue;
                slab |= 1u << e;
                P[e] = __ldg(prof + xe);
#pragma unroll
                for (int k = 0; k < TG; ++k) old[k][e] = J.slab[k][si[e]];
            }
        }
#pragma unroll
        for (int k = 0; k < TG; ++k) {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                v[e] = increment(p.dt, KIND == JOB_NORMAL ? normal_coef(a[e], b[e], k == J.diag) : a[e], d[e]);
                if (slab >> e & 1) {
                    const float sn = __fmul_rn(P[e], __fmaf_rn(P[e], old[k][e], v[e]));  // s <- P (P s + inc)
                    J.slab[k][si[e]] = sn;
                    v[e] = __fsub_rn(sn, old[k][e]);
                }
            }
            atomicAdd(reinterpret_cast<float4*>(tgt[k]) + i, make_float4(v[0], v[1], v[2], v[3]));
        }
    }
}

// the same by the tile's alignment and the kind of job
template <int NT, class LineOf>
__device__ __forceinline__ void x_quads_update(const PassParams& p, const PassJob& J, const float* bf, size_t q0, int line0,
                                               const XQuads& xq, int n, size_t off, size_t soff, LineOf line_of)
{
    if (J.kind == JOB_STORE && xq.on) x_quads_flat<NT, JOB_STORE, true>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    else if (J.kind == JOB_STORE) x_quads_flat<NT, JOB_STORE, false>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    else if (J.kind == JOB_SINGLE && xq.on) x_quads_flat<NT, JOB_SINGLE, true>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    else if (J.kind == JOB_SINGLE) x_quads_flat<NT, JOB_SINGLE, false>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    else if (xq.on) x_quads_flat<NT, JOB_NORMAL, true>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
    else x_quads_flat<NT, JOB_NORMAL, false>(p, J, bf, q0, line0, xq, n, off, soff, line_of);
}

// Epilogue of a tile of the x pass (lengths that are a multiple of 16): item by
// item, the next item's coefficients in flight; every access is a whole quad,
// the split parts of the PML slabs included.
template <int N, int NT, int PER, bool TM, int KIND>
__device__ __forceinline__ void x_epilogue(const PassParams& p, const PassJob& J, float* bf, const float* nearp,
                                           uint32_t tm, int line0, int nl, int sim)
{
    constexpr int LINES = 2 * PAIRS, ITEMS = LINES * N / 4, TG = KIND == JOB_NORMAL ? 3 : 1;
    const int tid = threadIdx.x;
    const size_t cell0 = (size_t)line0 * N, off = (size_t)sim * p.fstride + cell0;
    const float *co0 = J.coef[0] + cell0, *co1 = J.coef[1] + cell0;
    float* tgt[TG];
#pragma unroll
    for (int k = 0; k < TG; ++k) tgt[k] = J.tgt[k] + off;
    const float dt = p.dt;
    const int S = p.S;
    const size_t s0 = (size_t)sim * p.sstride + (size_t)line0 * S;
    const float* prof = J.stag ? p.ps : p.pc;
    float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0;
    auto coefs = [&](int it) {
        if (KIND == JOB_STORE || (ITEMS % NT != 0 && it >= ITEMS)) return;
        int r, xx;
        x_item<N>(it, &r, &xx);
        if (r >= nl || !ES_INB(p, cell0 + r * N + xx + 3, p.ext_c)) return;
        c0 = __ldg(reinterpret_cast<const float4*>(co0 + r * N + xx));
        if (KIND == JOB_NORMAL) c1 = __ldg(reinterpret_cast<const float4*>(co1 + r * N + xx));
    };
    coefs(tid);
#pragma unroll 1
    for (int i = 0; i < PER; ++i) {
        const int it = tid + i * NT;
        if (ITEMS % NT != 0 && it >= ITEMS) break;
        int r, xx;
        x_item<N>(it, &r, &xx);
        float n[4];
        if constexpr (TM) {
            tmem_ld<4>(tm + (uint32_t)(4 * i), n);
        } else {
            const float4 v = reinterpret_cast<const float4*>(nearp)[it];
            n[0] = v.x;
            n[1] = v.y;
            n[2] = v.z;
            n[3] = v.w;
        }
        const float4 d0 = c0, d1 = c1;
        if (i + 1 < PER) coefs(it + NT);
        if (r >= nl || !ES_INB(p, off + r * N + xx + 3, p.ext_f)) continue;
        float* f = bf + x_at<N>(xx, r);
        float d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = __fadd_rn(f[e * LINES], n[e]);
        const unsigned o = r * N + xx;
        if (KIND == JOB_STORE) {
            *reinterpret_cast<float4*>(tgt[0] + o) = make_float4(d[0], d[1], d[2], d[3]);
            continue;
        }
        const float a[4] = {d0.x, d0.y, d0.z, d0.w}, b[4] = {d1.x, d1.y, d1.z, d1.w};
        const bool slab = p.L > 0 && (xx < p.L || xx + 3 >= N - 1 - p.L);
        float4 P, old[TG];
        size_t so = 0;
        if (slab) {  // the quad's split parts (storage whole quads wide, slab_width)
            so = s0 + (size_t)r * S + (xx < p.L ? xx : xx - N + S);
            if (!ES_INB(p, so + 3, p.ext_s)) continue;
            P = __ldg(reinterpret_cast<const float4*>(prof + xx));
#pragma unroll
            for (int k = 0; k < TG; ++k) old[k] = *reinterpret_cast<const float4*>(J.slab[k] + so);
        }
#pragma unroll
        for (int k = 0; k < TG; ++k) {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                v[e] = increment(dt, KIND == JOB_NORMAL ? normal_coef(a[e], b[e], k == J.diag) : a[e], d[e]);
            if (slab) {
                const float P4[4] = {P.x, P.y, P.z, P.w}, s4[4] = {old[k].x, old[k].y, old[k].z, old[k].w};
                float n4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    n4[e] = __fmul_rn(P4[e], __fmaf_rn(P4[e], s4[e], v[e]));  // s <- P (P s + inc)
                    if (in_slab(xx + e, N, p.L)) v[e] = __fsub_rn(n4[e], s4[e]);
                }
                *reinterpret_cast<float4*>(J.slab[k] + so) = make_float4(n4[0], n4[1], n4[2], n4[3]);
            }
            atomicAdd(reinterpret_cast<float4*>(tgt[k] + o), make_float4(v[0], v[1], v[2], v[3]));
        }
    }
}

// x pass for lengths that are a multiple of 16, persistent as the y and z
// passes: a tile is 32 consecutive x-lines (line = y + ny z), one contiguous
// block of memory, which arrives as it is (raw) while the previous tile is
// worked on.  Items (four consecutive cells of a line) form the near parts
// along their line and turn the tile around into the FFT's [position][pencil]
// rows; at the end they read the far parts back from the turned-around rows, so
// every access to memory is four consecutive cells of 4 (or 8) lines per warp.
template <int RA, int RB, int RC, int T>
__global__ void __launch_bounds__(pass_threads<T>(), pass_min_blocks<RA, RB, RC, T>())
pass_x(const __grid_constant__ PassParams p, int ntiles)
{
    using C = CoreOf<RA, RB, RC, T>;
    constexpr int N = C::N, RN = N / T, NT = T * PAIRS;
    constexpr bool TM = near_in_tmem<N, T>();
    constexpr int LINES = 2 * PAIRS;
    constexpr int ITEMS = LINES * N / 4, PER = (ITEMS + NT - 1) / NT;  // items, and per thread
    static_assert(!TM || ITEMS % NT == 0, "tensor memory is read by whole warps");
    extern __shared__ __align__(16) float2 smem[];
    __shared__ uint32_t tmem_slot;
    float* raw = reinterpret_cast<float*>(smem);  // the tile as it is in memory
    float2* buf = smem + N * PAIRS;               // turned around: the FFT's rows
    float* nearp = reinterpret_cast<float*>(buf + N * PAIRS);  // near parts, item by item (not TM)
    float2* s_tw = buf + N * PAIRS + (TM ? 0 : N * PAIRS);
    float2* s_hp = s_tw + N;
    float2* s_hm = s_hp + N;
    float* bf = reinterpret_cast<float*>(buf);
    const int tid = threadIdx.x;
    const int c = tid % PAIRS, j = tid / PAIRS;
    uint32_t tm = 0;
    if (TM) {  // before dependents may launch (see pass_strided)
        if (tid < 32) tmem_alloc(&tmem_slot, tmem_columns<N, T>());
        __syncthreads();
        tm = tmem_slot + ((uint32_t)(tid / 32 % 4) << 21) + (uint32_t)(tid / 128 * 2 * RN);
    }
    pdl_begin(p.pdl);
    // the first pass of a fused time step advances the step counter
    if (p.step_counter && blockIdx.x == 0 && tid == 0) *p.step_counter += 1;
    const int nlines = p.ny * p.nz, total = ntiles * p.njobs;
    auto decode = [&](int w, int* sim) {  // first line of a tile
        w %= ntiles;
        *sim = p.nsim > 1 ? w % p.nsim : 0;
        return (p.nsim > 1 ? w / p.nsim : w) * LINES;
    };
    auto stage = [&](int w) {
        int sim;
        const int line0 = decode(w, &sim);
        const int nf = min(LINES, nlines - line0) * N;
        const size_t q = (size_t)sim * p.fstride + (size_t)line0 * N;
        const float* src = p.job[w / ntiles].src + q;
#pragma unroll 4
        for (int f = 4 * tid; f < LINES * N; f += 4 * NT) {
            const bool ok = f < nf && ES_INB(p, q + f + 3, p.ext_f);
            cp_async<16>(raw + f, ok ? src + f : src, ok);
        }
    };
    stage(blockIdx.x);
    for (int i = tid; i < N; i += NT) {
        s_tw[i] = __ldg(p.tw + i);
        s_hp[i] = __ldg(p.hp + i);
        s_hm[i] = __ldg(p.hm + i);
    }
    bool waited = p.pdl != 1;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        const PassJob& J = p.job[w / ntiles];
        int sim;
        const int line0 = decode(w, &sim), nl = min(LINES, nlines - line0);
        cp_async_commit_wait_all();
        __syncthreads();  // the tile is there; the previous tile's rows are no longer read
        // the tile's coefficient and slab lines (contiguous) into L2
        if (J.coef[0]) {
            const size_t q = (size_t)line0 * N, end = (size_t)nlines * N;
            for (int i = tid; i < N; i += NT)
                if (q + (size_t)i * 32 < end) {
                    prefetch_l2(J.coef[0] + q + (size_t)i * 32);
                    if (J.coef[1]) prefetch_l2(J.coef[1] + q + (size_t)i * 32);
                }
            if (p.L > 0) {
                const int S = p.S, ns = nl * S;
                const size_t s0 = (size_t)sim * p.sstride + (size_t)line0 * S;
                for (int f = 32 * tid; f < ns; f += 32 * NT) {
                    prefetch_l2(J.slab[0] + s0 + f);
                    if (J.coef[1]) {
                        prefetch_l2(J.slab[1] + s0 + f);
                        prefetch_l2(J.slab[2] + s0 + f);
                    }
                }
            }
        }
        // near parts along the lines, and the turn into the FFT's rows
        auto items = [&](auto sign) {
            constexpr int OFS = near_ofs(decltype(sign)::value);
            // x = xx - 8 .. xx + 11 in five chunks (wrapped along the line); the taps of the four
            // outputs reach xx + OFS .. xx + 3 + OFS + NEAR_TAPS - 1
            static_assert(8 + OFS >= 0 && 8 + 3 + OFS + NEAR_TAPS - 1 < 20, "near taps outside the window");
#pragma unroll 2
            for (int i = 0; i < PER; ++i) {
                const int it = tid + i * NT;
                if (ITEMS % NT != 0 && it >= ITEMS) break;
                int r, xx;
                x_item<N>(it, &r, &xx);
                const float* ln = raw + r * N;
                float v[20];
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    if (4 * m + 3 < 8 + OFS || 4 * m > 8 + 3 + OFS + NEAR_TAPS - 1) continue;  // chunk unused
                    int x0 = xx - 8 + 4 * m;
                    if (m < 2) x0 = x0 < 0 ? x0 + N : x0;
                    if (m > 2) x0 = x0 >= N ? x0 - N : x0;
                    const float4 f = *reinterpret_cast<const float4*>(ln + x0);
                    v[4 * m] = f.x;
                    v[4 * m + 1] = f.y;
                    v[4 * m + 2] = f.z;
                    v[4 * m + 3] = f.w;
                }
                float* d = bf + x_at<N>(xx, r);  // rows xx .. xx + 3 share the exchange
#pragma unroll
                for (int e = 0; e < 4; ++e) d[e * LINES] = v[8 + e];
                // outputs xx, xx + 1 and xx + 2, xx + 3 as packed pairs
                float2 s01 = make_float2(0.f, 0.f), s23 = make_float2(0.f, 0.f);
#pragma unroll
                for (int t = 0; t < NEAR_TAPS; ++t) {
                    const float2 g = rep2(J.g[t]);
                    s01 = fma2(g, make_float2(v[8 + OFS + t], v[9 + OFS + t]), s01);
                    s23 = fma2(g, make_float2(v[10 + OFS + t], v[11 + OFS + t]), s23);
                }
                if constexpr (TM) {
                    const float s[4] = {s01.x, s01.y, s23.x, s23.y};
                    tmem_st<4>(tm + (uint32_t)(4 * i), s);
                } else {
                    reinterpret_cast<float4*>(nearp)[it] = make_float4(s01.x, s01.y, s23.x, s23.y);
                }
            }
        };
        if (J.sign > 0) items(std::integral_constant<int, 1>{});
        else items(std::integral_constant<int, -1>{});
        __syncthreads();  // the rows are there; the raw tile has been read
        if (w + (int)gridDim.x < total) stage(w + gridDim.x);
        auto at = [&](int e) { return e * PAIRS + (c ^ x_swz<N>(e)); };
        {
            float2 a[C::MA][RA];
            C::stageA(a, j, [&](int e) { return buf[at(e)]; });
            __syncthreads();  // the turned-around rows have been read
            C::stageA_store(a, buf, j, c);
            __syncthreads();
            C::middle(buf, s_tw, J.sign > 0 ? s_hp : s_hm, j, c);
            __syncthreads();
            C::stageA_inv(buf, s_tw, a, j, c);
            __syncthreads();  // the FFT's rows have been read
            C::results(a, j, [&](int e, float2 v) { buf[at(e)] = make_float2(v.x, -v.y); });
        }
        if (TM) tmem_st_wait();
        __syncthreads();  // the far parts are there
        if (!waited) {
            pdl_wait();  // the previous pass's updates of the targets come first
            waited = true;
        }
        if (J.kind == JOB_STORE) x_epilogue<N, NT, PER, TM, JOB_STORE>(p, J, bf, nearp, tm, line0, nl, sim);
        else if (J.kind == JOB_SINGLE) x_epilogue<N, NT, PER, TM, JOB_SINGLE>(p, J, bf, nearp, tm, line0, nl, sim);
        else x_epilogue<N, NT, PER, TM, JOB_NORMAL>(p, J, bf, nearp, tm, line0, nl, sim);
    }
    if (TM) {
        __syncthreads();
        if (tid < 32) tmem_free(tmem_slot, tmem_columns<N, T>());
    }
}

// x pass for other lengths: blockIdx.x = tile of 32 consecutive x-lines,
// blockIdx.y = job.  After the inverse transform the derivatives are turned
// around through shared memory into memory order, and a thread updates four
// consecutive cells with 16-byte accesses from the targets' first 16-byte
// boundary on (x_quads).
template <int RA, int RB, int RC, int T>
__global__ void __launch_bounds__(pass_threads<T>(), pass_min_blocks<RA, RB, RC, T>(1250))
pass_x_any(const __grid_constant__ PassParams p)
{
    using C = CoreOf<RA, RB, RC, T>;
    constexpr int N = C::N, RN = N / T, NT = T * PAIRS;
    constexpr int LINES = 2 * PAIRS;
    extern __shared__ float2 smem[];
    float2* buf = smem;
    float2* nearp = buf + N * PAIRS;
    float2* s_tw = nearp + N * PAIRS;
    float2* s_h = s_tw + N;
    float* bf = reinterpret_cast<float*>(buf);
    const int tid = threadIdx.x;
    const int c = tid % PAIRS, j = tid / PAIRS;
    const PassJob& J = p.job[blockIdx.y];
    pdl_begin(p.pdl);
    // the first pass of a fused time step advances the step counter
    if (p.step_counter && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *p.step_counter += 1;
    const int nlines = p.ny * p.nz;
    const int sim = blockIdx.x % p.nsim;
    const size_t off = (size_t)sim * p.fstride, soff = (size_t)sim * p.sstride;
    const int line0 = (blockIdx.x / p.nsim) * LINES;
    const int nl = min(LINES, nlines - line0);
    const float* src = J.src + off;
    constexpr int XB = (N + 7) / 8, CELLS = LINES * XB * 8;
#pragma unroll
    for (int i = 0; i < (CELLS + NT - 1) / NT; ++i) {
        const int it = tid + i * NT;
        if (CELLS % NT != 0 && it >= CELLS) break;
        const int r = 4 * ((it >> 5) & 7) + ((it >> 3) & 3), xx = 8 * (it >> 8) + (it & 7);
        if (xx >= N) continue;
        const bool ok = r < nl && ES_INB(p, off + (size_t)(line0 + r) * N + xx, p.ext_f);
        cp_async<4>(bf + x_at<N>(xx, r), ok ? src + (size_t)(line0 + r) * N + xx : src, ok);
    }
    // the tile's coefficient lines (contiguous, N lines of 128 bytes) into L2
    if (J.coef[0]) {
        for (int i = tid; i < N; i += NT) {
            const size_t o = (size_t)line0 * N + (size_t)i * 32;
            if (o < (size_t)nlines * N) {
                prefetch_l2(J.coef[0] + o);
                if (J.coef[1]) prefetch_l2(J.coef[1] + o);
            }
        }
    }
    load_tables<N>(p, J, s_tw, s_h, tid, NT);
    cp_async_commit_wait_all();
    __syncthreads();
    auto at = [&](int e) { return e * PAIRS + (c ^ x_swz<N>(e)); };
    near_part<N, RN>(
        J, j, [&](int e) { return buf[at(e)]; }, [&](int q, float2 s) { nearp[at(RN * j + q)] = s; });
    float2 a[C::MA][RA];
    C::stageA(a, j, [&](int e) { return buf[at(e)]; });
    __syncthreads();  // the staged rows have been read; the near parts are visible
    C::stageA_store(a, buf, j, c);
    __syncthreads();
    C::middle(buf, s_tw, s_h, j, c);
    __syncthreads();
    C::stageA_inv(buf, s_tw, a, j, c);
    __syncthreads();  // the FFT rows have been read
    C::results(a, j, [&](int e, float2 v) {
        const float2 s = nearp[at(e)];
        float* o = bf + (2 * c) * N + e;  // lines 2c, 2c + 1 in memory order
        o[0] = __fadd_rn(v.x, s.x);
        o[N] = __fsub_rn(s.y, v.y);
    });
    __syncthreads();
    if (p.pdl == 1) pdl_wait();
    const size_t q0 = (size_t)line0 * N;
    const int nf = nl * N;
    const XQuads xq = x_quads(J, off, q0, nf);
    auto line_of = [](int f) { return f / N; };
    x_quads_update<NT>(p, J, bf, q0, line0, xq, N, off, soff, line_of);
    // what is left: the cells before the first chunk and past the last one
    for (int i = tid; i < nf - 4 * xq.nq; i += NT) {
        const int f = i < xq.h ? i : i + 4 * xq.nq, r = f / N, x = f - r * N, line = line0 + r;
        epilogue_one(p, J, q0 + f, x, x, line % p.ny, line / p.ny, bf[f], off, soff);
    }
}

}  // namespace es
