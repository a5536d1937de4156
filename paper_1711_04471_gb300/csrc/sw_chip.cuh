// 2DSW steps of a grid that fits on the chip (Sec. 6.2 of arXiv:1711.04471:
// dyn -> shapiro -> update): all steps of a call in one cooperative launch.
//
// A CTA (one per SM) owns a tile of tw x th cells and holds it with a halo
// of 2T cells on every side: H, eta, u, v of a thread's cells in registers,
// what neighbours read in shared memory.  It advances the whole region T
// steps (the valid part shrinks by two cells a step), then the tiles
// exchange: each publishes the cells within 2T of its own edge in global
// memory and reads its halo from there.  A published cell is one 16-byte
// word {eta, u, v, number of the exchange}, written and read as a single
// 128-bit access, so a reader polls the word itself and no flag, fence or
// barrier lies between two SMs.  Words alternate between two arrays; a tile
// publishes exchange k + 2 only after it has read exchange k + 1 from its
// neighbours, which they wrote after reading its exchange k.
//
// Each step is three barrier-separated phases over the region, as in
// sw_tile_kernel, with fewer operations: a face's flux is formed once, with
// its velocity; a cell publishes its eta* already multiplied by its wet
// mask, beside the mask; and the phases are branch-free, so that a thread's
// cells overlap.  Every rounding is the streaming kernel's, so
// the states are bitwise the same.  (Four cells of a row per thread with
// packed FP32 operations was slower: 3.2 us per step at 500x500.)
//
// What bounds it: the way of a word from SM to SM (about 1 us per exchange)
// on small grids, the issue slots and shared-memory wavefronts of the phases
// on large ones.  us per step, the kernel that the autotuner chose before,
// this one: 100x100 1.18, 0.65; all wet 500x500 2.54, 2.05; 15 % dry 700x700
// 4.98, 3.72 (untuned, the launches took 10 us and more); today's launches,
// this one: 800x800 6.7, 4.2 (all wet 5.9, 4.0); 900x900 7.1, 5.7 (6.4, 5.7).
#pragma once

#include "sw_kernels.cuh"

namespace gbsw {

constexpr int SWC_THREADS = 512;
constexpr int SWC_MAX_T = 4;
constexpr int SWC_GUARD = 2048;        // most columns of a region
constexpr int SWC_ARRAYS = 6;          // shared FP32 arrays of a region
constexpr int SWC_MAX_PER = 14;        // cells of a thread (13 and 14 spill a few bytes; with 15 and 16 the launches are faster)
constexpr long long SWC_WAIT_CYCLES = 4000000000LL;  // budget of a wait: about 2 s

// How a grid is cut: cx x cy tiles of tw x th cells (the last ones smaller),
// T steps between exchanges, `per` cells per thread; cx = 0: it does not fit.
struct SWChipPlan {
    int cx, cy, tw, th, T, per;
};

__device__ __forceinline__ uint4 swc_load(const uint4 *p)
{
    unsigned long long lo, hi;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}

__device__ __forceinline__ void swc_store(uint4 *p, float a, float b, float c, unsigned epoch)
{
    const unsigned long long lo = (unsigned long long)__float_as_uint(a) | ((unsigned long long)__float_as_uint(b) << 32);
    const unsigned long long hi = (unsigned long long)__float_as_uint(c) | ((unsigned long long)epoch << 32);
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n"
                 ::"l"(p), "l"(lo), "l"(hi) : "memory");
}

// nsteps steps from (eta_in, u_in, v_in) to (eta_out, u_out, v_out).  pub:
// two arrays of ny x nx words (NULL with a single tile); epoch0: number of
// the last exchange of earlier launches; wait: clock budget of a wait for
// another tile's word.  Cooperative launch: grid (cx, cy),
// block SWC_THREADS, SWC_ARRAYS x PER x SWC_THREADS + 2 SWC_GUARD floats of
// dynamic shared memory.
template <int PER>
__global__ void __launch_bounds__(SWC_THREADS, 1)
sw_chip_kernel(SWDev p, SWChipPlan P, int nsteps, unsigned epoch0, long long wait, uint4 *pub, int *status,
               const float *__restrict__ H, const float *__restrict__ eta_in, const float *__restrict__ u_in,
               const float *__restrict__ v_in, float *__restrict__ eta_out, float *__restrict__ u_out,
               float *__restrict__ v_out)
{
    constexpr int NC = PER * SWC_THREADS;
    constexpr bool FREG = PER <= 7;  // a cell's own fluxes wait in registers, else they are read back
    extern __shared__ float swc_smem[];
    // depth and elevation; fluxes through the east and north faces; masked
    // eta* and wet mask in pairs, and a row's worth of slack.  The rows below an
    // array's first and above its last one are read from what lies there (the
    // array before, the array after, the slack) and not used.
    float *const hh = swc_smem, *const e = hh + NC, *const ff = e + NC, *const gg = ff + NC;
    float2 *const we = reinterpret_cast<float2 *>(gg + NC);
    const int tid = threadIdx.x, T = P.T, halo = 2 * T;
    const int x0 = blockIdx.x * P.tw - halo, y0 = blockIdx.y * P.th - halo;
    const int tw = min(P.tw, p.nx - (int)blockIdx.x * P.tw), th = min(P.th, p.ny - (int)blockIdx.y * P.th);
    const int LW = tw + 2 * halo, LH = th + 2 * halo;  // LW LH <= NC
    const float hmin = p.hmin;
    const long long extent = (long long)p.ny * p.pitch, words = (long long)p.ny * p.nx;
    (void)extent;
    (void)words;
    constexpr unsigned F_CELL = 1u, F_EAST = 2u, F_NORTH = 4u, F_INNER = 8u, F_STORE = 16u, F_HALO = 32u, F_PUB = 64u;
    constexpr unsigned F_WET = 128u;  // wet at the start of the step
    float re[PER], ru[PER], rv[PER], rH[PER], rf[FREG ? PER : 1], rg[FREG ? PER : 1];
    unsigned m[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int q = tid + k * SWC_THREADS, ly = q / LW, lx = q - ly * LW;
        const int gx = x0 + lx, gy = y0 + ly;
        unsigned f = 0;
        re[k] = ru[k] = rv[k] = rH[k] = 0.0f;
        if (ly < LH) {
            f = F_CELL;
            if (lx + 1 < LW && gx >= 0 && gx < p.nx - 1) f |= F_EAST;
            if (ly + 1 < LH && gy >= 0 && gy < p.ny - 1) f |= F_NORTH;
            if (lx > 0 && lx + 1 < LW && ly > 0 && ly + 1 < LH) f |= F_INNER;
            const long long g = (long long)gy * p.pitch + gx;
            if (gx >= 0 && gx < p.nx && gy >= 0 && gy < p.ny && GBSW_INBOUNDS(g, extent, &g_sw_bounds)) {
                const bool own = lx >= halo && lx < halo + tw && ly >= halo && ly < halo + th;
                f |= own ? F_STORE : F_HALO;
                if (own && (lx < 2 * halo || lx >= tw || ly < 2 * halo || ly >= th)) f |= F_PUB;
                rH[k] = __ldg(H + g);
                re[k] = __ldg(eta_in + g);
                ru[k] = __ldg(u_in + g);
                rv[k] = __ldg(v_in + g);
            }
        }
        e[q] = re[k];
        hh[q] = __fadd_rn(rH[k], re[k]);
        m[k] = f;
    }
    __syncthreads();
    unsigned epoch = epoch0;
    for (int left = nsteps; left > 0;) {
        // a single tile has nothing to exchange (and no `pub`)
        const int n = gridDim.x * gridDim.y == 1 ? left : min(left, T);
        left -= n;
        for (int t = 0; t < n; ++t) {
            // Cells outside the inner region compute on whatever lies there and
            // keep their value.  Momentum predictor and flux of the east and
            // north faces of each cell
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int q = tid + k * SWC_THREADS;
                const float h = __fadd_rn(rH[k], re[k]), he = hh[q + 1], hn = hh[q + LW];
                const bool wc = h > hmin, east = m[k] & F_EAST, north = m[k] & F_NORTH;
                float a, b;
                ru[k] = sw_face(sw_predict(ru[k], p.gdt_dx, e[q + 1], re[k]), wc && east, he > hmin && east, &a, &b);
                const float f = __fmaf_rn(a, h, __fmul_rn(b, he));
                rv[k] = sw_face(sw_predict(rv[k], p.gdt_dy, e[q + LW], re[k]), wc && north, hn > hmin && north, &a, &b);
                const float g = __fmaf_rn(a, h, __fmul_rn(b, hn));
                ff[q] = f;
                gg[q] = g;
                if (FREG) {
                    rf[FREG ? k : 0] = f;
                    rg[FREG ? k : 0] = g;
                }
            }
            __syncthreads();
            // continuity; the masked eta* and the mask
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int q = tid + k * SWC_THREADS;
                const bool wc = __fadd_rn(rH[k], re[k]) > hmin;
                const float f = FREG ? rf[FREG ? k : 0] : ff[q], g = FREG ? rg[FREG ? k : 0] : gg[q];
                const float es = __fsub_rn(re[k], __fmaf_rn(p.dt_dx, __fsub_rn(f, ff[q - 1]),
                                                            __fmul_rn(p.dt_dy, __fsub_rn(g, gg[q - LW]))));
                re[k] = m[k] & F_INNER ? es : re[k];
                const float w = wc ? 1.0f : 0.0f;
                we[q] = make_float2(__fmul_rn(w, re[k]), w);
                m[k] = (m[k] & ~F_WET) | (wc ? F_WET : 0u);
            }
            __syncthreads();
            // masked Shapiro filter on wet cells; the next step's depth
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int q = tid + k * SWC_THREADS;
                const float2 ae = we[q + 1], aw = we[q - 1], an = we[q + LW], as = we[q - LW];
                const float sum = __fadd_rn(__fadd_rn(ae.x, aw.x), __fadd_rn(an.x, as.x));
                const float cnt = (ae.y + aw.y) + (an.y + as.y);  // small integers: exact
                const float out = __fmaf_rn(p.q, sum, __fmul_rn(__fsub_rn(1.0f, __fmul_rn(p.q, cnt)), re[k]));
                re[k] = (m[k] & (F_INNER | F_WET)) == (F_INNER | F_WET) ? out : re[k];
                e[q] = re[k];
                hh[q] = __fadd_rn(rH[k], re[k]);
            }
            __syncthreads();
        }
        if (left == 0) break;
        // exchange
        ++epoch;
        uint4 *const w = pub + (epoch & 1u) * (size_t)p.ny * p.nx;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (m[k] & F_PUB) {
                const int q = tid + k * SWC_THREADS, ly = q / LW;
                const long long g = (long long)(y0 + ly) * p.nx + x0 + q - ly * LW;
                if (GBSW_INBOUNDS(g, words, &g_sw_bounds)) swc_store(w + g, re[k], ru[k], rv[k], epoch);
            }
        bool late = false;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (m[k] & F_HALO) {
                const int q = tid + k * SWC_THREADS, ly = q / LW;
                const long long g = (long long)(y0 + ly) * p.nx + x0 + q - ly * LW;
                if (!GBSW_INBOUNDS(g, words, &g_sw_bounds)) continue;
                uint4 v = swc_load(w + g);
                if (v.w != epoch) {
                    const long long t0 = clock64();
                    do {
                        if (clock64() - t0 > wait) {
                            late = true;
                            break;
                        }
                        v = swc_load(w + g);
                    } while (v.w != epoch);
                }
                re[k] = __uint_as_float(v.x);
                ru[k] = __uint_as_float(v.y);
                rv[k] = __uint_as_float(v.z);
                e[q] = re[k];
                hh[q] = __fadd_rn(rH[k], re[k]);
            }
        if (__syncthreads_or(late)) {
            if (tid == 0) set_device_status(status, DEV_TIMEOUT);
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k)
        if (m[k] & F_STORE) {
            const int q = tid + k * SWC_THREADS, ly = q / LW;
            const long long g = (long long)(y0 + ly) * p.pitch + x0 + q - ly * LW;
            eta_out[g] = re[k];
            u_out[g] = ru[k];
            v_out[g] = rv[k];
        }
}

}  // namespace gbsw
