// Streaming, temporally blocked 2DSW kernel (Sec. 6.2 of arXiv:1711.04471:
// dyn -> shapiro -> update, fused over T time steps).
//
// Work decomposition.  A CTA of SWS_THREADS threads owns a strip of
// SWS_THREADS grid columns (one column per thread), of which the middle
// W = SWS_THREADS - 4T are written back (2 columns of halo per fused step
// on each side), and a segment of rows [r0, r1).  It marches up the strip
// one row per iteration.  Time level t -> t+1 is a pipeline stage: stage t
// receives a row of level t and emits the level-(t+1) row two rows below
// it (the y-radius of one step's dependency cone).  Stage t+1 consumes
// what stage t emitted in the previous iteration; stage t works 3t rows
// behind stage 0 and the strip's output row trails the input row by 3T-1.
//
// Each thread keeps the y-neighbours of its own column in registers (the
// rolling window below); x-neighbours go through per-stage shared-memory
// line buffers.  Global memory is touched once per fused launch: level 0
// rows (eta, u, v, H) are loaded four rows ahead, level T rows are stored.
//
// One step on row n (level t -> t+1), with h = H + eta, w = h > hmin:
//   u'(n), F(n)     = face(u - g dt/dx (eta_e - eta_c))   (needs eta, h at (x+1, n))
//   v'(n-1), G(n-1) = face(v - g dt/dy (eta(n) - eta(n-1)))
//   eta*(n-1) = eta - dt/dx (F - F_w) - dt/dy (G - G_s)   (F_w(n-1): the line of the last iteration)
//   eta+(n-2) = Shapiro filter of w eta*                  (the lines' row n-2: the last iteration's)
// Only (eta, h) are read in the iteration that publishes them, so one
// barrier per row is enough: a line slot is rewritten two iterations after
// it was filled, with a barrier between its last read and the rewrite.
//
// Bound by issued instructions (86 per cell and step, 58 % of the issue
// slots) and the latencies that four warps per scheduler leave open.  Each
// face's flux is formed once, w eta* travels with w, loads and stores are
// predicated, a wall is a wet threshold of infinity.  With three barriers
// per row, branches and the fluxes formed on both sides of every face a step
// took (T = 3, 15 % of the cells dry) at 4096x4096 74.6 us, now 61.0; 2000x2000
// 23.6, 18.7; 1237x1501 15.0, 10.7 (all wet: 17.1 and 9.6 for the last two).
#pragma once

#include <type_traits>

#include "sw_kernels.cuh"

namespace gbsw {

constexpr int SWS_THREADS = 128;   // strip width (threads = columns)
constexpr int SWS_PAD = 1;         // one guard column on each side of a line buffer
constexpr int SWS_LINE = SWS_THREADS + 2 * SWS_PAD;

// Rolling per-stage window of one column (registers).
struct SWStageRegs {
    float eta1, h1, v1;  // level-t row n-1
    float H1, H2;        // still-water depth at rows n-1, n-2
    float F1, G2;        // fluxes: F at row n-1, G at row n-2
    float up1, up2, vp2; // u' at rows n-1, n-2, v' at row n-2
    float es2;           // eta* at row n-2
    float we2, we3;      // w eta* at rows n-2, n-3
    float w1, w2, w3;    // w at rows n-1, n-2, n-3
};

// A row of one column handed from a stage to the next (or loaded / stored).
struct SWRow {
    float eta, u, v, H;
};

// Per-stage shared line buffers.
struct SWStageLines {
    float2 eh[2][SWS_LINE];  // eta, h of the incoming row
    float2 ws[2][SWS_LINE];  // w eta*, w
    float F[2][SWS_LINE];    // flux through the east faces
};

// Loads of the level-0 rows: through the read-only path when the inputs
// cannot change during the kernel (one fused launch), through L2 only
// (coherent across SMs) inside the persistent ensemble kernel, where other
// CTAs rewrite the buffers between levels.
enum class SWLoad { ReadOnly, L2 };

// *ptr if ok, else 0; and *ptr = v if ok: one predicated access, no branch.
template <SWLoad LP>
__device__ __forceinline__ float sw_load(const float *ptr, bool ok)
{
    float v;
    if constexpr (LP == SWLoad::ReadOnly)
        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n mov.f32 %0, 0f00000000;\n @p ld.global.nc.f32 %0, [%1];\n}"
                     : "=f"(v) : "l"(ptr), "r"((unsigned)ok));
    else
        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n mov.f32 %0, 0f00000000;\n @p ld.global.cg.f32 %0, [%1];\n}"
                     : "=f"(v) : "l"(ptr), "r"((unsigned)ok) : "memory");
    return v;
}

__device__ __forceinline__ void sw_store(float *ptr, float v, bool ok)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p st.global.f32 [%0], %1;\n}"
                 :: "l"(ptr), "f"(v), "r"((unsigned)ok) : "memory");
}

// One (strip, row segment) work item: T fused steps of the columns of
// strip `strip` (SWS_THREADS wide, W = SWS_THREADS - 4T written) for output
// rows [r0, r1).  All threads of the CTA must call it together.
template <int T, SWLoad LP>
__device__ __forceinline__ void sw_stream_tile(const SWDev &p, int strip, int r0, int r1,
                                               const float *__restrict__ H, const float *__restrict__ eta_in,
                                               const float *__restrict__ u_in, const float *__restrict__ v_in,
                                               float *__restrict__ eta_out, float *__restrict__ u_out,
                                               float *__restrict__ v_out, SWStageLines *lines)
{
    constexpr int W = SWS_THREADS - 4 * T;
    const int x = threadIdx.x;
    const int c = x + SWS_PAD;                      // index in a line buffer
    const int gi = strip * W - 2 * T + x;           // grid column of this thread
    const bool col_in = gi >= 0 && gi < p.nx;
    const bool owned = x >= 2 * T && x < 2 * T + W && col_in;
    const bool u_open = gi >= 0 && gi < p.nx - 1;   // not a wall face
    __syncthreads();  // the line buffers may still be in use by the previous work item

    // zero the guard columns once (they only feed discarded halo columns)
    if (x < 2 * T) {
        const int st = x >> 1;
        const int side = (x & 1) ? SWS_LINE - 1 : 0;
        for (int k = 0; k < 2; ++k) {
            lines[st].eh[k][side] = lines[st].ws[k][side] = make_float2(0.0f, 0.0f);
            lines[st].F[k][side] = 0.0f;
        }
    }

    const float hmin = p.hmin, inf = __int_as_float(0x7f800000);
    const float hmin_u = u_open ? hmin : inf;  // wet threshold of the east face: nothing is above it at a wall
    SWStageRegs R[T];
    SWRow mail[T];  // mail[t]: level-(t+1) row emitted by stage t last iteration
#pragma unroll
    for (int t = 0; t < T; ++t) {
        R[t] = SWStageRegs{};
        mail[t] = SWRow{0, 0, 0, 0};
    }

    const long long extent = (long long)p.ny * p.pitch;  // elements of each field of this grid
    auto load_row = [&](int n) {
        const long long g = (long long)n * p.pitch + gi;
        const bool ok = col_in & ((unsigned)n < (unsigned)p.ny) && GBSW_INBOUNDS(g, extent, &g_sw_bounds);
        SWRow r;
        r.eta = sw_load<LP>(eta_in + g, ok);
        r.u = sw_load<LP>(u_in + g, ok);
        r.v = sw_load<LP>(v_in + g, ok);
        r.H = sw_load<LP>(H + g, ok);
        return r;
    };

    // The row loop is unrolled by 4 so that every line slot and the shift of
    // the register window are resolved at compile time.
    const int n_first = (r0 - 2 * T) & ~3;    // first level-0 row that matters, rounded down
    const int n_last = r1 - 1 + 3 * T - 1;    // iteration that emits output row r1-1
    SWRow pre[4];  // the rows ahead: four cover the latency of a load from DRAM
#pragma unroll
    for (int k = 0; k < 4; ++k) pre[k] = load_row(n_first + k);

    auto iteration = [&](auto phase, int n4) {
        constexpr int P = decltype(phase)::value;  // n & 3
        const int n = n4 + P;
        SWRow in[T];
        in[0] = pre[P];
        pre[P] = load_row(n + 4);
#pragma unroll
        for (int t = 1; t < T; ++t) in[t] = mail[t - 1];

        // publish eta and h of the incoming row of every stage
        float hn[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int s0 = (P - 3 * t) & 1;  // slot of row m = n - 3t
            hn[t] = __fadd_rn(in[t].H, in[t].eta);
            lines[t].eh[s0][c] = make_float2(in[t].eta, hn[t]);
        }
        __syncthreads();
        // what the neighbour columns published, of all stages at once: the
        // stages' arithmetic interleaves between the loads and the stores
        float2 ee[T], ae[T], aw[T];
        float Fw[T], Fn[T], we[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int s0 = (P - 3 * t) & 1, s1 = s0 ^ 1;  // slots of row m (and m-2), of row m-1
            ee[t] = lines[t].eh[s0][c + 1];
            Fw[t] = lines[t].F[s1][c - 1];
            ae[t] = lines[t].ws[s0][c + 1];
            aw[t] = lines[t].ws[s0][c - 1];
        }
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int m = n - 3 * t;
            SWStageRegs &r = R[t];
            float a, b;
            // momentum predictor and fluxes: u'(m), F(m), v'(m-1), G(m-1)
            const float un = sw_face(sw_predict(in[t].u, p.gdt_dx, ee[t].x, in[t].eta), hn[t] > hmin_u,
                                     ee[t].y > hmin_u, &a, &b);
            Fn[t] = __fmaf_rn(a, hn[t], __fmul_rn(b, ee[t].y));
            const float hmin_v = (unsigned)(m - 1) < (unsigned)(p.ny - 1) ? hmin : inf;
            const float vn = sw_face(sw_predict(r.v1, p.gdt_dy, in[t].eta, r.eta1), r.h1 > hmin_v,
                                     hn[t] > hmin_v, &a, &b);
            const float Gn = __fmaf_rn(a, r.h1, __fmul_rn(b, hn[t]));
            // continuity: eta*(m-1)
            const float es = __fsub_rn(r.eta1, __fmaf_rn(p.dt_dx, __fsub_rn(r.F1, Fw[t]), __fmul_rn(p.dt_dy, __fsub_rn(Gn, r.G2))));
            we[t] = __fmul_rn(r.w1, es);
            // Shapiro filter: eta+(m-2); emit the level-(t+1) row m-2
            const float cnt = (ae[t].y + aw[t].y) + (r.w1 + r.w3);  // small integers: exact
            const float sum = __fadd_rn(__fadd_rn(ae[t].x, aw[t].x), __fadd_rn(we[t], r.we3));
            const float flt = __fmaf_rn(p.q, sum, __fmul_rn(__fsub_rn(1.0f, __fmul_rn(p.q, cnt)), r.es2));
            mail[t] = SWRow{r.w2 != 0.0f ? flt : r.es2, r.up2, r.vp2, r.H2};
            // roll the window
            r.eta1 = in[t].eta;
            r.h1 = hn[t];
            r.v1 = in[t].v;
            r.H2 = r.H1;
            r.H1 = in[t].H;
            r.F1 = Fn[t];
            r.G2 = Gn;
            r.up2 = r.up1;
            r.up1 = un;
            r.vp2 = vn;
            r.es2 = es;
            r.we3 = r.we2;
            r.we2 = we[t];
            r.w3 = r.w2;
            r.w2 = r.w1;
            r.w1 = hn[t] > hmin ? 1.0f : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const int s0 = (P - 3 * t) & 1, s1 = s0 ^ 1;
            lines[t].F[s0][c] = Fn[t];
            lines[t].ws[s1][c] = make_float2(we[t], R[t].w2);
        }
        // the last stage's row is final: level T at row n - 3T + 1
        const int out_row = n - 3 * T + 1;
        const long long g = (long long)out_row * p.pitch + gi;
        const bool ok = owned & ((unsigned)(out_row - r0) < (unsigned)(r1 - r0)) && GBSW_INBOUNDS(g, extent, &g_sw_bounds);
        sw_store(eta_out + g, mail[T - 1].eta, ok);
        sw_store(u_out + g, mail[T - 1].u, ok);
        sw_store(v_out + g, mail[T - 1].v, ok);
    };

#pragma unroll 1
    for (int n4 = n_first; n4 <= n_last; n4 += 4) {
        iteration(std::integral_constant<int, 0>{}, n4);
        iteration(std::integral_constant<int, 1>{}, n4);
        iteration(std::integral_constant<int, 2>{}, n4);
        iteration(std::integral_constant<int, 3>{}, n4);
    }
}

// One fused launch of depth T over a single grid.  grid (strips, segments),
// block SWS_THREADS; rows_per_cta rows per segment.
template <int T>
__global__ void __launch_bounds__(SWS_THREADS)
sw_stream_kernel(SWDev p, int rows_per_cta, const float *__restrict__ H, const float *__restrict__ eta_in,
                 const float *__restrict__ u_in, const float *__restrict__ v_in, float *__restrict__ eta_out,
                 float *__restrict__ u_out, float *__restrict__ v_out)
{
    __shared__ SWStageLines lines[T];
    const int r0 = blockIdx.y * rows_per_cta;
    if (r0 >= p.ny) return;
    const int r1 = min(p.ny, r0 + rows_per_cta);
    sw_stream_tile<T, SWLoad::ReadOnly>(p, blockIdx.x, r0, r1, H, eta_in, u_in, v_in, eta_out, u_out, v_out, lines);
}

}  // namespace gbsw
