// FP64 2DSW time step (Sec. 6.2 of arXiv:1711.04471) as the paper's three
// map kernels per step: the predictor "dyn" split into its momentum part
// (faces) and its continuity part (cells), then the first-order Shapiro
// filter, with the velocity/state update folded into buffer swaps.
//
// Every operation is written out in the order of the method as stated in
// include/gbsw.h and rounded as written (explicit round-to-nearest FP64
// intrinsics, no multiply-add contraction):
//   u'   = u - ((g dt) (eta_e - eta_c)) / dx, masked by the wet/dry face rule
//   F    = max(u', 0) h_behind + min(u', 0) h_ahead      (two products, one sum)
//   eta* = eta - dt ((F_e - F_w) / dx + (G_n - G_s) / dy)
//   eta+ = (1 - q n) eta*_c + q s on wet cells, q = eps / 4, where n counts
//          the wet neighbours and s sums their eta* in the order east, west,
//          north, south; dry cells keep eta*
// so that the state is a deterministic function of the inputs, bit for bit
// the same on every launch shape.  FP32 is the fast path (sw_step); this
// variant exists for precision: it is the method in FP64 end to end.
//
// What bounds it.  An FP64 instruction takes this GPU as long as 64 FP32 or
// integer ones, so the kernels are written for few FP64 instructions (31 per
// cell and step, against about 110 for the formulas as they stand) with the
// same roundings:
//   - the depth h = H + eta is formed once per cell and step and kept;
//   - a face's flux is formed once, with its velocity (one of its two
//     products is a zero);
//   - comparisons are integer comparisons of the bit patterns;
//   - a division by dx or dy is a product with the rounded reciprocal and
//     one or two FMA corrections (s64_div), correctly rounded;
//   - 1 - q n comes from a table of five values.
// 700x501 cells, 15 % dry: 89 us per step with the formulas as they stand, 39 so;
// the FP64 pipe's floor for 31 instructions per cell is 17 us.
//
// Device layout: (ny + 2) rows of `pitch` doubles, cell (i, j) (1-based
// interior, 0 and n + 1 the halo ring) at j * pitch + i; u[j][i] and F[j][i]
// are the east face of cell (i, j) (i = 0 .. nx), v[j][i] and G[j][i] the
// north face (j = 0 .. ny).  Walls and the halo ring stay 0 (h = 0 reads as
// dry).
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "common.cuh"

struct gbsw_sw64 {
    gbsw_sw_params p;
    int pitch;
    cudaStream_t stream;
    double *H;                // (ny+2) x pitch
    double *eta, *u, *v;      // the state, updated in place
    double *F, *G;            // fluxes through the east and north faces
    double *h[2];             // depth H + eta at the start of the step ([cur]) and of the next one
    double *es;               // eta* of the step
    int cur;
    cudaGraphExec_t chunk[2]; // S64_CHUNK steps from h[0], h[1] as a graph
    double *partials, *result;
    double *h_result;         // pinned, 3 doubles
};

namespace {

constexpr int S64_THREADS = 128;
constexpr int S64_VOL_BLOCKS = 512;

constexpr int S64_CHUNK = 16;  // steps per replayed graph (even: a chunk ends on the buffer it started from)

struct S64Dev {
    int nx, ny, pitch;
    double gdt;   // g * dt
    double dx, dy, dt;
    double q;     // eps / 4
    double hmin;
    double ydx, ydy;      // RN(1 / dx), RN(1 / dy)
    int ndx, ndy;         // corrections that s64_div needs (0: plain division)
    long long hmin_bits;  // of hmin (not negative)
    double coef[5];       // RN(1 - RN(q n))
};

constexpr long long S64_INF = 0x7ff0000000000000LL;

__device__ __forceinline__ bool s64_wet(const S64Dev &p, double h)  // h > hmin
{
    const long long b = __double_as_longlong(h);
    return b > p.hmin_bits && b <= S64_INF;
}
__device__ __forceinline__ bool s64_pos(double x)  // x > 0
{
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= S64_INF;
}
__device__ __forceinline__ bool s64_neg(double x)  // x < 0
{
    return s64_pos(__longlong_as_double(__double_as_longlong(x) ^ (1LL << 63)));
}
__device__ __forceinline__ int s64_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x / d rounded to nearest even, y = RN(1/d): q = RN(x y); if q is within one
// unit in the last place, its remainder is exact in one FMA and q + r y,
// rounded once, is the correctly rounded quotient (P. Markstein, "IA-64 and
// Elementary Functions", Prentice Hall 2000, ch. 8).  q is off by less than
// 1/2 unit (its own rounding) + 2 |1 - y d| 2^52 units, so n = 1 when
// |1 - y d| <= 2^-54, else a second correction follows the first.  Exponents
// at which a remainder could leave the normal range take the division.
__device__ __forceinline__ double s64_div(double x, double d, double y, int n)
{
    if (n > 0 && (unsigned)(s64_exponent(x) - 200) < 1600u) {
        double q = __dmul_rn(x, y);
        q = __fma_rn(__fma_rn(-q, d, x), y, q);
        if (n > 1) q = __fma_rn(__fma_rn(-q, d, x), y, q);
        return q;
    }
    if ((__double_as_longlong(x) << 1) == 0) return x;  // a zero
    return __ddiv_rn(x, d);
}

// Wet/dry face rule: a is the cell behind the face, b the cell ahead.
__device__ __forceinline__ double s64_mask(double vel, bool wet_a, bool wet_b)
{
    return (wet_a && wet_b) || (wet_a && s64_pos(vel)) || (wet_b && s64_neg(vel)) ? vel : 0.0;
}

// Upwind volume flux max(vel, 0) h_a + min(vel, 0) h_b through a face: one of
// the products is a zero unless the other depth is not finite.
__device__ __forceinline__ double s64_flux(double vel, double h_a, double h_b)
{
    const bool pos = s64_pos(vel), neg = s64_neg(vel);
    if (s64_exponent(h_a) == 0x7ff || s64_exponent(h_b) == 0x7ff)
        return __dadd_rn(__dmul_rn(pos ? vel : 0.0, h_a), __dmul_rn(neg ? vel : 0.0, h_b));
    return pos || neg ? __dmul_rn(vel, pos ? h_a : h_b) : 0.0;
}

// The kernels of a step follow one another as programmatic launches: each
// may be scheduled while the one before drains, and reads nothing before
// that one has completed.
__device__ __forceinline__ void s64_wait()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch of the kernels that set up and read the state: columns x rows, a
// block taking rows y, y + gridDim.y, ... (a grid has at most 65535 in y).
dim3 s64_rows_grid(int columns, int rows)
{
    return dim3(gbsw::ceil_div(columns, S64_THREADS), std::min(rows, 65535));
}

// h = H + eta on the interior (the initial state).
__global__ void __launch_bounds__(S64_THREADS)
sw64_depth_kernel(S64Dev p, const double *H, const double *eta, double *h)
{
    const int i = blockIdx.x * S64_THREADS + threadIdx.x + 1;
    if (i > p.nx) return;
    for (int j = blockIdx.y + 1; j <= p.ny; j += gridDim.y) {
        const long long c = (long long)j * p.pitch + i;
        h[c] = __dadd_rn(H[c], eta[c]);
    }
}

// Map 1 ("dyn", momentum): u' and its flux on the east faces i = 1 .. nx-1,
// v' and its flux on the north faces j = 1 .. ny-1 (wall faces stay 0).
// Launch of the three maps: grid (ceil(nx / S64_THREADS), ny), block S64_THREADS.
__global__ void __launch_bounds__(S64_THREADS)
sw64_momentum_kernel(S64Dev p, const double *eta, const double *h, double *u, double *v, double *F, double *G)
{
    s64_wait();
    const int i = blockIdx.x * S64_THREADS + threadIdx.x + 1, j = blockIdx.y + 1;
    if (i > p.nx) return;
    const long long c = (long long)j * p.pitch + i, n = c + p.pitch;
    const double ec = eta[c], hc = h[c];
    const bool wc = s64_wet(p, hc);
    if (i < p.nx) {
        const double he = h[c + 1];
        const double pred = __dsub_rn(u[c], s64_div(__dmul_rn(p.gdt, __dsub_rn(eta[c + 1], ec)), p.dx, p.ydx, p.ndx));
        const double vel = s64_mask(pred, wc, s64_wet(p, he));
        u[c] = vel;
        F[c] = s64_flux(vel, hc, he);
    }
    if (j < p.ny) {
        const double hn = h[n];
        const double pred = __dsub_rn(v[c], s64_div(__dmul_rn(p.gdt, __dsub_rn(eta[n], ec)), p.dy, p.ydy, p.ndy));
        const double vel = s64_mask(pred, wc, s64_wet(p, hn));
        v[c] = vel;
        G[c] = s64_flux(vel, hc, hn);
    }
}

// Map 2 ("dyn", continuity): eta* on every interior cell.
__global__ void __launch_bounds__(S64_THREADS)
sw64_continuity_kernel(S64Dev p, const double *eta, const double *F, const double *G, double *es)
{
    s64_wait();
    const int i = blockIdx.x * S64_THREADS + threadIdx.x + 1, j = blockIdx.y + 1;
    if (i > p.nx) return;
    const long long c = (long long)j * p.pitch + i;
    const double div = __dadd_rn(s64_div(__dsub_rn(F[c], F[c - 1]), p.dx, p.ydx, p.ndx),
                                 s64_div(__dsub_rn(G[c], G[c - p.pitch]), p.dy, p.ydy, p.ndy));
    es[c] = __dsub_rn(eta[c], __dmul_rn(p.dt, div));
}

// Map 3 ("shapiro"): masked 5-point filter of eta* on wet cells (wet mask
// of the start of the step), and the depth of the next step.
__global__ void __launch_bounds__(S64_THREADS)
sw64_shapiro_kernel(S64Dev p, const double *H, const double *h, const double *es, double *eta, double *h_next)
{
    s64_wait();
    const int i = blockIdx.x * S64_THREADS + threadIdx.x + 1, j = blockIdx.y + 1;
    if (i > p.nx) return;
    const long long c = (long long)j * p.pitch + i;
    double out = es[c];
    if (s64_wet(p, h[c])) {
        const long long nb[4] = {c + 1, c - 1, c + p.pitch, c - p.pitch};
        int count = 0;
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (s64_wet(p, h[nb[k]])) {
                const double e = es[nb[k]];
                sum = count ? __dadd_rn(sum, e) : e;
                ++count;
            }
        const double coef = count == 4 ? p.coef[4] : count == 3 ? p.coef[3] : count == 2 ? p.coef[2]
                          : count == 1 ? p.coef[1] : p.coef[0];
        out = __dadd_rn(__dmul_rn(coef, out), __dmul_rn(p.q, sum));
    }
    eta[c] = out;
    h_next[c] = __dadd_rn(H[c], out);
}

// Rows 0 .. rows-1 of `width` elements from `src` (row pitch p.pitch) packed into dst.
__global__ void __launch_bounds__(S64_THREADS)
sw64_pack_kernel(S64Dev p, const double *src, int width, int rows, double *dst)
{
    const int i = blockIdx.x * S64_THREADS + threadIdx.x;
    if (i >= width) return;
    for (int j = blockIdx.y; j < rows; j += gridDim.y) dst[(size_t)j * width + i] = src[(size_t)j * p.pitch + i];
}

// Wet mask of the state as bytes.
__global__ void __launch_bounds__(S64_THREADS)
sw64_wet_kernel(S64Dev p, const double *h, uint8_t *wet)
{
    const int i = blockIdx.x * S64_THREADS + threadIdx.x;
    if (i >= p.nx) return;
    for (int j = blockIdx.y; j < p.ny; j += gridDim.y)
        wet[(size_t)j * p.nx + i] = h[(size_t)(j + 1) * p.pitch + i + 1] > p.hmin;
}

// FP64 volume partials over rows b, b + S64_VOL_BLOCKS, ... (fixed order).
__global__ void __launch_bounds__(256)
sw64_volume_partial_kernel(S64Dev p, const double *__restrict__ H, const double *__restrict__ eta,
                           double *__restrict__ partials)
{
    __shared__ double red[256 / 32];
    double s = 0.0, sw = 0.0, bad = 0.0;
    for (int j = blockIdx.x + 1; j <= p.ny; j += S64_VOL_BLOCKS)
        for (int i = threadIdx.x + 1; i <= p.nx; i += blockDim.x) {
            const long long c = (long long)j * p.pitch + i;
            if (!isfinite(eta[c])) bad += 1.0;
            const double h = __dadd_rn(H[c], eta[c]);
            s += h;
            if (h > p.hmin) sw += h;
        }
    s = gbsw::block_sum_f64<256 / 32>(s, red);
    sw = gbsw::block_sum_f64<256 / 32>(sw, red);
    bad = gbsw::block_sum_f64<256 / 32>(bad, red);
    if (threadIdx.x == 0) {
        partials[3 * blockIdx.x] = s;
        partials[3 * blockIdx.x + 1] = sw;
        partials[3 * blockIdx.x + 2] = bad;
    }
}

__global__ void __launch_bounds__(256)
sw64_volume_final_kernel(S64Dev p, const double *__restrict__ partials, double *__restrict__ out)
{
    __shared__ double red[256 / 32];
    double s = 0.0, sw = 0.0, bad = 0.0;
    for (int b = threadIdx.x; b < S64_VOL_BLOCKS; b += blockDim.x) {
        s += partials[3 * b];
        sw += partials[3 * b + 1];
        bad += partials[3 * b + 2];
    }
    s = gbsw::block_sum_f64<256 / 32>(s, red);
    sw = gbsw::block_sum_f64<256 / 32>(sw, red);
    bad = gbsw::block_sum_f64<256 / 32>(bad, red);
    if (threadIdx.x == 0) {
        out[0] = __dmul_rn(__dmul_rn(s, p.dx), p.dy);
        out[1] = __dmul_rn(__dmul_rn(sw, p.dx), p.dy);
        out[2] = bad;
    }
}

S64Dev s64_dev(const gbsw_sw64 *s)
{
    S64Dev d;
    d.nx = s->p.nx;
    d.ny = s->p.ny;
    d.pitch = s->pitch;
    d.gdt = s->p.g * s->p.dt;
    d.dx = s->p.dx;
    d.dy = s->p.dy;
    d.dt = s->p.dt;
    d.q = 0.25 * s->p.eps;
    d.hmin = s->p.hmin + 0.0;  // + 0.0: -0 as 0
    memcpy(&d.hmin_bits, &d.hmin, sizeof(d.hmin));
    for (int n = 0; n < 5; ++n) {
        const volatile double qn = d.q * n;  // two roundings, as written
        d.coef[n] = 1.0 - qn;
    }
    auto corrections = [](double x, double *y) {
        *y = 1.0 / x;
        if (!(x > 0x1p-100 && x < 0x1p100)) return 0;
        return fabs(fma(-*y, x, 1.0)) <= 0x1p-54 ? 1 : 2;
    };
    d.ndx = corrections(d.dx, &d.ydx);
    d.ndy = corrections(d.dy, &d.ydy);
    return d;
}

// One step from depth buffer a, on stream st; after: the launch before this one is another step's.
cudaError_t s64_enqueue(const gbsw_sw64 *s, const S64Dev &d, int a, cudaStream_t st, bool after)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(gbsw::ceil_div(d.nx, S64_THREADS), d.ny);
    cfg.blockDim = dim3(S64_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = after ? attr : nullptr;
    cfg.numAttrs = after ? 1 : 0;
    const double *H = s->H, *h = s->h[a], *F = s->F, *G = s->G, *es = s->es, *eta = s->eta;
    cudaError_t e = cudaLaunchKernelEx(&cfg, sw64_momentum_kernel, d, eta, h, s->u, s->v, s->F, s->G);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, sw64_continuity_kernel, d, eta, F, G, s->es);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, sw64_shapiro_kernel, d, H, h, es, s->eta, s->h[1 - a]);
    return e;
}

// The graph of S64_CHUNK steps from depth buffer a (captured on a private stream).
cudaError_t s64_chunk(gbsw_sw64 *s, const S64Dev &d, int a)
{
    if (s->chunk[a]) return cudaSuccess;
    cudaStream_t cs = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t el = cudaSuccess;
        for (int k = 0; k < S64_CHUNK && el == cudaSuccess; ++k) el = s64_enqueue(s, d, (a + k) & 1, cs, k > 0);
        e = cudaStreamEndCapture(cs, &g);
        if (e == cudaSuccess) e = el;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&s->chunk[a], g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) s->chunk[a] = nullptr;
    return e;
}

}  // namespace

using namespace gbsw;

extern "C" {

void sw64_destroy(gbsw_sw64 *s)
{
    if (!s) return;
    cudaStreamSynchronize(s->stream);
    for (cudaGraphExec_t g : s->chunk)
        if (g) cudaGraphExecDestroy(g);
    double *bufs[] = {s->H, s->eta, s->u, s->v, s->F, s->G, s->h[0], s->h[1], s->es, s->partials, s->result};
    for (double *b : bufs) cudaFree(b);
    if (s->h_result) cudaFreeHost(s->h_result);
    delete s;
}

gbsw_status sw64_create(const gbsw_sw_params *params, const double *H, const double *eta0, void *stream,
                        gbsw_sw64 **out)
{
    if (!params || !H || !eta0 || !out) return GBSW_ERR_ARG;
    const gbsw_sw_params P = *params;
    if (P.nx < 2 || P.ny < 2 || P.nx > (1 << 20) || P.ny > (1 << 20)) return GBSW_ERR_ARG;
    if (!(P.dx > 0) || !(P.dy > 0) || !(P.dt > 0) || !(P.g > 0) || !(P.eps >= 0 && P.eps <= 1) ||
        !(P.hmin >= 0))
        return GBSW_ERR_ARG;
    const size_t n = (size_t)P.nx * (size_t)P.ny;
    std::vector<double> e(n);
    double hmax = 0.0;
    for (size_t k = 0; k < n; ++k) {
        if (!std::isfinite(H[k]) || !std::isfinite(eta0[k])) return GBSW_ERR_ARG;
        e[k] = eta0[k] < -H[k] ? -H[k] : eta0[k];
        hmax = std::max(hmax, H[k] + e[k]);
    }
    const double courant = sqrt(P.g * hmax) * P.dt * sqrt(1.0 / (P.dx * P.dx) + 1.0 / (P.dy * P.dy));
    if (courant > 1.0) return GBSW_ERR_CFL;
    if (fault_injected("alloc")) return GBSW_ERR_OOM;

    gbsw_sw64 *s = new (std::nothrow) gbsw_sw64();
    if (!s) return GBSW_ERR_OOM;
    s->p = P;
    s->pitch = (int)round_up((size_t)P.nx + 2, 16);
    s->stream = (cudaStream_t)stream;
    const size_t bytes = (size_t)s->pitch * (size_t)(P.ny + 2) * sizeof(double);
    double **fields[] = {&s->H, &s->eta, &s->u, &s->v, &s->F, &s->G, &s->h[0], &s->h[1], &s->es};
    for (double **f : fields) {
        cudaError_t err = cudaMalloc((void **)f, bytes);
        if (err == cudaSuccess) err = cudaMemsetAsync(*f, 0, bytes, s->stream);
        if (err != cudaSuccess) {
            record_cuda_error(err, "sw64_create", __FILE__, __LINE__);
            sw64_destroy(s);
            return err == cudaErrorMemoryAllocation ? GBSW_ERR_OOM : GBSW_ERR_CUDA;
        }
    }
    cudaError_t err = cudaMalloc((void **)&s->partials, 3 * S64_VOL_BLOCKS * sizeof(double));
    if (err == cudaSuccess) err = cudaMalloc((void **)&s->result, 3 * sizeof(double));
    if (err == cudaSuccess) err = cudaMallocHost((void **)&s->h_result, 3 * sizeof(double));
    // interior rows 1..ny, columns 1..nx of H and eta
    const size_t dp = (size_t)s->pitch * sizeof(double), hp = (size_t)P.nx * sizeof(double);
    if (err == cudaSuccess)
        err = cudaMemcpy2DAsync(s->H + s->pitch + 1, dp, H, hp, hp, P.ny, cudaMemcpyHostToDevice, s->stream);
    if (err == cudaSuccess)
        err = cudaMemcpy2DAsync(s->eta + s->pitch + 1, dp, e.data(), hp, hp, P.ny, cudaMemcpyHostToDevice, s->stream);
    if (err == cudaSuccess) {
        sw64_depth_kernel<<<s64_rows_grid(P.nx, P.ny), S64_THREADS, 0, s->stream>>>(s64_dev(s), s->H, s->eta, s->h[0]);
        err = cudaGetLastError();
    }
    if (err == cudaSuccess) err = cudaStreamSynchronize(s->stream);
    if (err != cudaSuccess) {
        record_cuda_error(err, "sw64_create", __FILE__, __LINE__);
        sw64_destroy(s);
        return err == cudaErrorMemoryAllocation ? GBSW_ERR_OOM : GBSW_ERR_CUDA;
    }
    *out = s;
    return GBSW_OK;
}

gbsw_status sw64_step(gbsw_sw64 *s, int nsteps)
{
    gbsw::NvtxRange nvtx_range("sw64_step");
    if (!s || nsteps < 0) return GBSW_ERR_ARG;
    const S64Dev d = s64_dev(s);
    int left = nsteps;
    cudaError_t e = cudaSuccess;
    for (; left >= S64_CHUNK && e == cudaSuccess; left -= S64_CHUNK) {
        e = s64_chunk(s, d, s->cur);
        if (e == cudaSuccess) e = cudaGraphLaunch(s->chunk[s->cur], s->stream);
    }
    for (int k = 0; k < left && e == cudaSuccess; ++k) {
        e = s64_enqueue(s, d, s->cur, s->stream, k > 0);
        if (e == cudaSuccess) s->cur = 1 - s->cur;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();  // reported here, not by the next call
        record_cuda_error(e, "sw64_step", __FILE__, __LINE__);
        return GBSW_ERR_CUDA;
    }
    return GBSW_OK;
}

gbsw_status sw64_volume(gbsw_sw64 *s, double *volume, double *wet_volume)
{
    if (!s) return GBSW_ERR_ARG;
    const S64Dev d = s64_dev(s);
    sw64_volume_partial_kernel<<<S64_VOL_BLOCKS, 256, 0, s->stream>>>(d, s->H, s->eta, s->partials);
    sw64_volume_final_kernel<<<1, 256, 0, s->stream>>>(d, s->partials, s->result);
    GBSW_LAUNCH_CHECK();
    GBSW_CUDA_TRY(cudaMemcpyAsync(s->h_result, s->result, 3 * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    GBSW_CUDA_TRY(cudaStreamSynchronize(s->stream));
    if (volume) *volume = s->h_result[0];
    if (wet_volume) *wet_volume = s->h_result[1];
    return s->h_result[2] > 0.0 ? GBSW_ERR_NONFINITE : GBSW_OK;
}

gbsw_status sw64_get_state(gbsw_sw64 *s, double *eta, double *u, double *v, uint8_t *wet)
{
    if (!s) return GBSW_ERR_ARG;
    const int nx = s->p.nx, ny = s->p.ny;
    // Each field is packed on the device (into es, which the next step writes
    // anew) and copied in one piece: a pitched copy into pageable memory goes
    // row by row.
    const S64Dev d = s64_dev(s);
    auto copy = [&](double *dst, const double *src, int width, int rows) -> gbsw_status {
        sw64_pack_kernel<<<s64_rows_grid(width, rows), S64_THREADS, 0, s->stream>>>(d, src, width, rows, s->es);
        GBSW_LAUNCH_CHECK();
        GBSW_CUDA_TRY(cudaMemcpyAsync(dst, s->es, (size_t)width * rows * sizeof(double), cudaMemcpyDeviceToHost,
                                      s->stream));
        return GBSW_OK;
    };
    gbsw_status st = GBSW_OK;
    if (eta) st = copy(eta, s->eta + s->pitch + 1, nx, ny);
    if (u && st == GBSW_OK) st = copy(u, s->u + s->pitch, nx + 1, ny);  // east faces i = 0..nx of rows 1..ny
    if (v && st == GBSW_OK) st = copy(v, s->v + 1, nx, ny + 1);         // north faces j = 0..ny of columns 1..nx
    if (st != GBSW_OK) return st;
    if (wet) {
        sw64_wet_kernel<<<s64_rows_grid(nx, ny), S64_THREADS, 0, s->stream>>>(d, s->h[s->cur], (uint8_t *)s->es);
        GBSW_LAUNCH_CHECK();
        GBSW_CUDA_TRY(cudaMemcpyAsync(wet, s->es, (size_t)nx * ny, cudaMemcpyDeviceToHost, s->stream));
    }
    GBSW_CUDA_TRY(cudaStreamSynchronize(s->stream));
    return GBSW_OK;
}

}  // extern "C"
