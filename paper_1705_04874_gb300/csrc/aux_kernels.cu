// Small kernels around the derivative passes: point-source injection
// (Sec. II-A: point sources at grid points), 4C receiver recording
// (Sec. II-A, Eq. (3); Sec. II-B), superposition of single-event traces
// (Sec. IV), a non-finite scan and slab initialisation.
#include <algorithm>

#include "es_internal.h"

namespace es {

// One thread walks every source in order, so sources sharing a cell add in a
// fixed order.  The step counter lives on the device so that one captured
// step can be replayed: the kernel that runs last in a step (`advance`)
// publishes the step index to `cur` for the recorder and increments it.
// The spatial-frequency Blackman window of one axis, W(m) = 0.42 + 0.5 cos(2 pi m / n)
// + 0.08 cos(4 pi m / n) over the signed wavenumber bins m (1 at m = 0, 0 at the
// Nyquist bin), has the inverse DFT 0.42 at offset 0, 0.25 at +-1, 0.04 at +-2
// and 0 elsewhere (n >= 5): the smoothed point source (Sec. II-A) is exactly the
// product of these three stencils around the source cell.
__constant__ float c_blackman5[5] = {0.04f, 0.25f, 0.42f, 0.25f, 0.04f};

// One block.  Thread 0 adds the point sources in order (deterministic); then
// every thread takes (source, stencil cell) pairs of the smoothed sources and
// adds with reductions (order free only where smoothed stencils of one
// simulation overlap); then thread 0 advances the step counter.
__global__ void inject_kernel(float* const* fields, long long fstride, const SourceDev* src, int nsrc, int kind,
                              int nx, int ny, int* counter, int* cur, int advance)
{
    const int n = *counter;
    if (threadIdx.x == 0) {
        for (int e = 0; e < nsrc; ++e) {
            const SourceDev s = src[e];
            if (s.kind != kind || s.smooth || n >= s.nw) continue;
            const float w = s.w[n];
            const long long q = (long long)s.sim * fstride + s.cell;
            if (kind == 0) {
                // moment tensor: stress component i gains M_i w[n] (Mxx Myy Mzz Mxy Mxz Myz)
                for (int c = 0; c < 6; ++c)
                    if (s.m[c] != 0.f) fields[SXX + c][q] = __fmaf_rn(s.m[c], w, fields[SXX + c][q]);
            } else {
                // point force: m[c] = dt f_c / (rho_c dx dy dz), folded on the host
                for (int c = 0; c < 3; ++c)
                    if (s.m[c] != 0.f) fields[VX + c][q] = __fmaf_rn(s.m[c], w, fields[VX + c][q]);
            }
        }
    }
    __syncthreads();
    if (kind == 0) {
        for (int it = threadIdx.x; it < nsrc * 125; it += blockDim.x) {
            const int e = it / 125, k = it % 125;
            const SourceDev& s = src[e];
            if (!s.smooth || s.kind != 0 || n >= s.nw) continue;
            const int dx = k % 5 - 2, dy = (k / 5) % 5 - 2, dz = k / 25 - 2;
            const float g = c_blackman5[dx + 2] * c_blackman5[dy + 2] * c_blackman5[dz + 2];
            const float w = s.w[n] * g;
            const long long q = (long long)s.sim * fstride + s.cell + dx + (long long)nx * (dy + (long long)ny * dz);
            for (int c = 0; c < 6; ++c)
                if (s.m[c] != 0.f) atomicAdd(fields[SXX + c] + q, s.m[c] * w);
        }
    }
    __syncthreads();
    if (advance && threadIdx.x == 0) {
        *cur = n;
        *counter = n + 1;
    }
}

cudaError_t launch_inject(float* const* fields, long long fstride, const SourceDev* src, int nsrc, int kind,
                          int nx, int ny, int* counter, int* cur, int advance, cudaStream_t st)
{
    inject_kernel<<<1, 256, 0, st>>>(fields, fstride, src, nsrc, kind, nx, ny, counter, cur, advance);
    return cudaGetLastError();
}

// Kelvin-Voigt source of the stress passes: w = a v - b vold, vold <- v, for
// the three velocity components ([c][sim][cell], n = cells x simulations each)
__global__ void visc_combine_kernel(float* const* fields, float* vold, float* w, size_t n, float a, float b)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float v = fields[VX + c][i];
            w[c * n + i] = a * v - b * vold[c * n + i];
            vold[c * n + i] = v;
        }
}

cudaError_t launch_visc_combine(float* const* fields, float* vold, float* w, size_t n, float a, float b,
                                cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const size_t blocks = std::min<size_t>((n + 255) / 256, 152 * 16);
    visc_combine_kernel<<<(unsigned)blocks, 256, 0, st>>>(fields, vold, w, n, a, b);
    return cudaGetLastError();
}

// Material coefficients of one cell per thread (Eq. (4) and the staggered
// averages of the model setup): lambda = rho cp^2 - 2 mu and mu = rho cs^2 at
// the cell, buoyancy 2 / (rho_i + rho_(i+1)) at the half-index point along
// each axis, and the edge shear moduli as the harmonic mean of the four
// surrounding mu (0 if any is 0, i.e. next to water); neighbours wrap
// periodically.  FP64 with explicitly rounded operations (no contraction),
// stored in FP32.
__device__ __forceinline__ double mu_of(const float* rho, const float* cs, size_t p)
{
    const double s = cs[p];
    return __dmul_rn(__dmul_rn(s, s), (double)rho[p]);
}

__device__ __forceinline__ double harmonic4(double a, double b, double c, double d)
{
    if (a == 0.0 || b == 0.0 || c == 0.0 || d == 0.0) return 0.0;
    const double s = __dadd_rn(__dadd_rn(__dadd_rn(__ddiv_rn(1.0, a), __ddiv_rn(1.0, b)), __ddiv_rn(1.0, c)),
                               __ddiv_rn(1.0, d));
    return __ddiv_rn(4.0, s);
}

__global__ void materials_kernel(const float* rho, const float* cp, const float* cs, int nx, int ny, int nz,
                                 MatPtrs out)
{
    const size_t n = (size_t)nx * ny * nz;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(q % nx), j = (int)((q / nx) % ny), k = (int)(q / ((size_t)nx * ny));
        const int ip = i + 1 == nx ? 0 : i + 1, jp = j + 1 == ny ? 0 : j + 1, kp = k + 1 == nz ? 0 : k + 1;
        auto at = [&](int ii, int jj, int kk) { return (size_t)ii + (size_t)nx * ((size_t)jj + (size_t)ny * kk); };
        const size_t qx = at(ip, j, k), qy = at(i, jp, k), qz = at(i, j, kp);
        const double r = rho[q], c = cp[q];
        const double mu = mu_of(rho, cs, q);
        out.p[M_LAM][q] = __double2float_rn(__dsub_rn(__dmul_rn(__dmul_rn(c, c), r), __dmul_rn(2.0, mu)));
        out.p[M_MU][q] = __double2float_rn(mu);
        out.p[M_BX][q] = __double2float_rn(__ddiv_rn(2.0, __dadd_rn(r, (double)rho[qx])));
        out.p[M_BY][q] = __double2float_rn(__ddiv_rn(2.0, __dadd_rn(r, (double)rho[qy])));
        out.p[M_BZ][q] = __double2float_rn(__ddiv_rn(2.0, __dadd_rn(r, (double)rho[qz])));
        const double mx = mu_of(rho, cs, qx), my = mu_of(rho, cs, qy), mz = mu_of(rho, cs, qz);
        out.p[M_MUXY][q] = __double2float_rn(harmonic4(mu, mx, my, mu_of(rho, cs, at(ip, jp, k))));
        out.p[M_MUXZ][q] = __double2float_rn(harmonic4(mu, mx, mz, mu_of(rho, cs, at(ip, j, kp))));
        out.p[M_MUYZ][q] = __double2float_rn(harmonic4(mu, my, mz, mu_of(rho, cs, at(i, jp, kp))));
    }
}

cudaError_t launch_materials(const float* rho, const float* cp, const float* cs, int nx, int ny, int nz,
                             const MatPtrs& out, cudaStream_t st)
{
    const size_t n = (size_t)nx * ny * nz;
    if (n == 0) return cudaSuccess;
    const size_t blocks = std::min<size_t>((n + 255) / 256, 152 * 32);
    materials_kernel<<<(unsigned)blocks, 256, 0, st>>>(rho, cp, cs, nx, ny, nz, out);
    return cudaGetLastError();
}

__global__ void fill_kernel(float* p, size_t n, float v)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) p[i] = v;
}

cudaError_t launch_fill(float* p, size_t n, float v, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const size_t blocks = std::min<size_t>((n + 255) / 256, 4096);
    fill_kernel<<<(unsigned)blocks, 256, 0, st>>>(p, n, v);
    return cudaGetLastError();
}

// rec[n - start][sim][c][r]: sample n of component c (p, vx, vy, vz) of
// simulation sim at receiver r
__global__ void record_kernel(float* const* fields, long long fstride, int nsim, const long long* rcv_cell, int n_rcv,
                              const int* cur, long long start, float* rec)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_rcv * nsim) return;
    const int r = i % n_rcv, sim = i / n_rcv;
    const long long q = (long long)sim * fstride + rcv_cell[r];
    const size_t row = ((size_t)(*cur - start) * nsim + sim) * 4 * n_rcv;
    const float s = __fadd_rn(__fadd_rn(fields[SXX][q], fields[SYY][q]), fields[SZZ][q]);
    rec[row + r] = __fdiv_rn(-s, 3.f);  // Eq. (3)
    rec[row + n_rcv + r] = fields[VX][q];
    rec[row + 2 * (size_t)n_rcv + r] = fields[VY][q];
    rec[row + 3 * (size_t)n_rcv + r] = fields[VZ][q];
}

cudaError_t launch_record(float* const* fields, long long fstride, int nsim, const long long* rcv_cell, int n_rcv,
                          const int* cur, long long start, float* rec, cudaStream_t st)
{
    if (n_rcv <= 0) return cudaSuccess;
    const int n = n_rcv * nsim;
    record_kernel<<<(n + 127) / 128, 128, 0, st>>>(fields, fstride, nsim, rcv_cell, n_rcv, cur, start, rec);
    return cudaGetLastError();
}

// [rows][cols] -> [cols][rows] through a 32 x 32 shared tile
__global__ void transpose_kernel(const float* in, int rows, int cols, float* out)
{
    __shared__ float tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[i][threadIdx.x] = in[(size_t)r * cols + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (r < rows && c < cols) out[(size_t)c * rows + r] = tile[threadIdx.x][i];
    }
}

cudaError_t launch_transpose_traces(const float* rec, int nt, int cols, float* out, cudaStream_t st)
{
    dim3 grid((cols + 31) / 32, (nt + 31) / 32), block(32, 8);
    transpose_kernel<<<grid, block, 0, st>>>(rec, nt, cols, out);
    return cudaGetLastError();
}

// gather[row][t] = sum_e amp_e traces[src_e][row][t - k_e], rows = 4 n_rcv, in
// FP32 with the events in order (one multiply-add per event and sample).
//
// A warp owns 32 R consecutive output samples of one row, R per thread (lane +
// 32 i), and walks the events once: per event one uniform test of how its trace
// overlaps the span (not at all, wholly, partly), then R coalesced loads and R
// multiply-adds, so the event's bookkeeping is paid once per 32 R samples.  What
// bounds it is the L2 -> SM traffic: an event's trace is read at its own shift,
// 4 bytes per event and sample (a trace itself comes from DRAM about once: the
// rows in flight fit in L2).  Events reach shared memory in chunks of SUP_CHUNK,
// so any number of them fits without changing the order of the sum.
// Small gathers do not have the warps to hide an event's load behind other
// warps: there the events that overlap the span go U at a time, the loads of all
// of them before the first multiply-add.
// 64 sources x 1024 receivers x 2000 samples, 300 events into 4666 samples (one
// GB300): 1.28 ms (1.44 ms with the call around it); one sample per thread with
// a test, an address and three shared loads per event and sample took 4.54 (4.70).
constexpr int SUP_CHUNK = 1024, SUP_WARPS = 8;

template <int R, int U>
__global__ void __launch_bounds__(32 * SUP_WARPS) superpose_kernel(const float* traces, long long rows, int nt,
                                                                   const int* ev_src, const float* ev_amp,
                                                                   const int* ev_shift, int n_events, int n_out,
                                                                   int spans, float* gather)
{
    struct Event {
        long long ofs;  // of the event's trace in row 0, at sample -k
        int k;
        float amp;
    };
    __shared__ __align__(16) Event ev[SUP_CHUNK + (U > 1 ? 1 : 0)];
    const long long unit = (long long)blockIdx.x * SUP_WARPS + threadIdx.x / 32;  // row-major: consecutive warps share a row
    const long long row = unit / spans;
    const bool active = row < rows;
    const int t0 = (int)(unit - row * spans) * 32 * R, lane = threadIdx.x % 32;
    const float* base = traces + row * nt + t0 + lane;
    float acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = 0.f;
    for (int e0 = 0; e0 < n_events; e0 += SUP_CHUNK) {
        const int ne = min(SUP_CHUNK, n_events - e0);
        __syncthreads();  // the previous chunk is no longer read
        for (int i = threadIdx.x; i < ne; i += 32 * SUP_WARPS) {
            // a shift past either end of the window: no overlap with any span
            int k = ev_shift[e0 + i];
            if (k <= -nt || k > n_out) k = n_out;
            ev[i].ofs = (long long)ev_src[e0 + i] * rows * nt - k;
            ev[i].k = k;
            ev[i].amp = ev_amp[e0 + i];
        }
        // what fills up a group: an event past the window (row 0 of source 0, at a shift of n_out)
        if (U > 1 && threadIdx.x == 0) ev[SUP_CHUNK] = {-(long long)n_out, n_out, 0.f};
        __syncthreads();
        if (!active) continue;
        if constexpr (U > 1) {
#pragma unroll 1
            for (int g = 0; g < ne; g += 32) {  // a lane tests one event of 32, the warp walks those that overlap
                const int k0 = t0 - (g + lane < ne ? ev[g + lane].k : n_out);
                unsigned todo = __ballot_sync(0xffffffffu, g + lane < ne && k0 < nt && k0 + 32 * R > 0);
#pragma unroll 1
                while (todo) {
                    float x[U][R], amp[U];
                    bool in[U][R];
#pragma unroll
                    for (int j = 0; j < U; ++j) {
                        const Event v = ev[todo ? g + __ffs(todo) - 1 : SUP_CHUNK];
                        todo &= todo - 1;
                        const int u = t0 - v.k + lane;
                        amp[j] = v.amp;
#pragma unroll
                        for (int i = 0; i < R; ++i) {
                            in[j][i] = u + 32 * i >= 0 && u + 32 * i < nt;
                            x[j][i] = in[j][i] ? __ldg(base + v.ofs + 32 * i) : 0.f;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < U; ++j)
#pragma unroll
                        for (int i = 0; i < R; ++i) acc[i] = in[j][i] ? __fmaf_rn(amp[j], x[j][i], acc[i]) : acc[i];
                }
            }
            continue;
        }
#pragma unroll 2
        for (int e = 0; e < ne; ++e) {
            const Event v = ev[e];
            const int u = t0 - v.k;  // trace sample of the span's first output sample
            if (u >= nt || u + 32 * R <= 0) continue;
            const float* x = base + v.ofs;
            if (u >= 0 && u + 32 * R <= nt) {
#pragma unroll
                for (int i = 0; i < R; ++i) acc[i] = __fmaf_rn(v.amp, __ldg(x + 32 * i), acc[i]);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int ui = u + lane + 32 * i;
                    if (ui >= 0 && ui < nt) acc[i] = __fmaf_rn(v.amp, __ldg(x + 32 * i), acc[i]);
                }
            }
        }
    }
    if (!active) return;
    float* out = gather + row * n_out + t0 + lane;
#pragma unroll
    for (int i = 0; i < R; ++i)
        if (t0 + lane + 32 * i < n_out) out[32 * i] = acc[i];
}

template <int R, int U>
static cudaError_t launch_superpose_r(const float* traces, int n_rcv, int nt, const int* ev_src, const float* ev_amp,
                                      const int* ev_shift, int n_events, int n_out, float* gather, cudaStream_t st)
{
    const long long rows = 4LL * n_rcv, spans = (n_out + 32LL * R - 1) / (32 * R);
    const long long blocks = (rows * spans + SUP_WARPS - 1) / SUP_WARPS;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    superpose_kernel<R, U><<<(unsigned)blocks, 32 * SUP_WARPS, 0, st>>>(traces, rows, nt, ev_src, ev_amp, ev_shift,
                                                                    n_events, n_out, (int)spans, gather);
    return cudaGetLastError();
}

cudaError_t launch_superpose(const float* traces, int n_src, int n_rcv, int nt, const int* ev_src,
                             const float* ev_amp, const int* ev_shift, int n_events, int n_out, float* gather,
                             cudaStream_t st)
{
    (void)n_src;
    // us a call by output samples (one GB300, 300 events; one sample per thread in brackets).  R = 8 and
    // 4: 19.1 M 1282 and 1270 (4541), 12.3 M with short traces 297 and 372 (2597), 5.1 M 229 and 272 (1173), 1.28 M
    // 101 and 115 (325), 1.02 M 63 and 74 (250), 307 K 102 and 89 (112): below about a million the longer spans
    // leave SMs idle.  Below half a million R = 4 does too; R = 4, and R = 2 with the events eight at a time:
    // 384 K 59 and 55 (118), 307 K 89 and 64 (112), 96 K 51 and 45 (55), 32 K 86 and 42 (42), 8 K with 60,000
    // events 3732 and 1577 (2672); 1.02 M 75 and 77.
    if (4LL * n_rcv * n_out >= 1 << 20)
        return launch_superpose_r<8, 1>(traces, n_rcv, nt, ev_src, ev_amp, ev_shift, n_events, n_out, gather, st);
    if (4LL * n_rcv * n_out >= 1 << 19)
        return launch_superpose_r<4, 1>(traces, n_rcv, nt, ev_src, ev_amp, ev_shift, n_events, n_out, gather, st);
    return launch_superpose_r<2, 8>(traces, n_rcv, nt, ev_src, ev_amp, ev_shift, n_events, n_out, gather, st);
}

// flag |= 1 if any field value is NaN or infinite
__global__ void nonfinite_kernel(float* const* fields, size_t n, int* flag)
{
    int bad = 0;
    for (int f = 0; f < NFIELD; ++f) {
        const float* a = fields[f];
        for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
            bad |= !isfinite(a[i]);
    }
    bad = __syncthreads_or(bad);
    if (bad && threadIdx.x == 0) atomicOr(flag, 1);
}

cudaError_t launch_nonfinite(float* const* fields, size_t n, int* flag, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    nonfinite_kernel<<<sms * 4, 256, 0, st>>>(fields, n, flag);
    return cudaGetLastError();
}

// slab[cell in slab] = copy ? total[cell] : 0 (0 in an x slab's unused cells)
__global__ void fill_slab_kernel(const float* total, float* slab, int axis, int nx, int ny, int nz, int L,
                                 int copy)
{
    const int S = slab_width(axis, L);
    const int n = axis == 0 ? nx : (axis == 1 ? ny : nz);
    const size_t cnt = (size_t)nx * ny * nz / n * S;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < cnt; i += (size_t)gridDim.x * blockDim.x) {
        int x, y, z, sp;
        if (axis == 0) { sp = (int)(i % S); size_t l = i / S; y = (int)(l % ny); z = (int)(l / ny); x = 0; }
        else if (axis == 1) { x = (int)(i % nx); size_t l = i / nx; sp = (int)(l % S); z = (int)(l / S); y = 0; }
        else { x = (int)(i % nx); size_t l = i / nx; y = (int)(l % ny); sp = (int)(l / ny); z = 0; }
        const int pos = sp < L ? sp : sp - S + n;
        if (sp >= L && pos < n - 1 - L) {
            slab[i] = 0.f;
            continue;
        }
        if (axis == 0) x = pos; else if (axis == 1) y = pos; else z = pos;
        slab[i] = copy ? total[(size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * z)] : 0.f;
    }
}

cudaError_t launch_fill_slab(const float* total, float* slab, int axis, int nx, int ny, int nz, int L, int copy,
                             cudaStream_t st)
{
    fill_slab_kernel<<<1024, 256, 0, st>>>(total, slab, axis, nx, ny, nz, L, copy);
    return cudaGetLastError();
}

}  // namespace es
