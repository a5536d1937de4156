// The whole pressure solve in one cooperative launch, for grids whose SOR
// correction fits in the shared memory of all SMs together ("press",
// Sec. 6.3.1 of arXiv:1711.04471).
//
// Decomposition.  The (j, k) rows of the grid are cut into py x pz
// rectangles, one CTA (and one SM) each; a CTA keeps the correction e of
// both colours of its rows in shared memory for the whole solve, in the
// slot order of the colour arrays (16-byte groups of four slots, no
// padding), and the residual r beside it when both fit (RSMEM), else r
// stays in the global colour arrays and streams in from L2.  Rows on the
// rectangle's rim are also published in global memory, where the up to four
// neighbouring CTAs read them.  sort_plan (poisson.cu) picks the cut.
//
// Register tiles (sort_register_sweeps; up to 4 groups per thread, about
// 2.4 M cells on 152 SMs).  What bounds them is the way of a value from one
// SM to another, about 1 us.  Each published value travels with an epoch
// (the number of the half-sweep that wrote it) in one 64-bit element: a
// reader polls the value itself until it carries the epoch, so no flag,
// fence or barrier lies between the two SMs.  A value is overwritten
// (half-sweep h + 2) only after its reader's own value of h + 1, written
// after that read, has been consumed.
//
// Larger tiles (sort_sweeps).  A half-sweep costs the shared-memory
// wavefronts and the issue slots of its updates.  Inside the rim a thread
// owns two adjacent rows of one group and marches in z: the other colour's
// vectors of the two rows serve as x neighbours, as each other's y
// neighbours and, one plane later or earlier, as z neighbours, so an update
// of four cells reads two vectors of the other colour, its own and r, and
// writes one; FP32 operations run two to an instruction.  The rim comes
// first and is published with one flag count per warp; a neighbour looks at
// the flags in the middle of its march and reads the rows ahead.
//
// Every wait is bounded by a clock
// budget; a wait that gives up records DEV_TIMEOUT and the CTA returns.
//
// Measured, us per iteration (half-sweep launches, this kernel):
// 256x256x128 16.9, 13.0; 300x300x90 18.3, 14.2; 256x128x64 8.8, 5.2;
// 160x96x64 10.0, 3.2; 72x48x40 5.4, 2.2; 16x16x12 4.5, 0.75 (one CTA).
//
// Checks.  A register tile whose FP64 pressure and right-hand side fit in
// shared memory too (psm, about 2 M cells) runs the whole solve in one
// launch: the FP64 residual of a 160x96x64 grid and its way through the grid
// barriers take about 20 us, three kernels and a loop node took 50. Larger
// grids keep the residual as a kernel of its own in a graph's loop: it is
// bound by the FP64 pipe and wants the warps that this kernel's registers
// do not allow (0.20 ms against 0.13 at 256x256x128).
//
// Arithmetic.  Every update is that of sor_sweep_kernel, operation by
// operation, so the iterates are bitwise the same; the residual norms are
// summed in another (fixed) order.
#pragma once

#include <type_traits>

#include "poisson.cuh"

namespace gbsw {

constexpr int SORT_THREADS = 384;           // of a tile of any size: 168 registers a thread
constexpr int SORT_SMALL_THREADS = 512;     // of a tile whose cells live in registers
constexpr int SORT_HALO = 4;                // halo groups that a thread of such a tile fetches at most
constexpr int SORT_TILE_BYTES = 768;        // header of the dynamic shared memory
constexpr int SORT_KINDS = 16;              // kinds of group by their diagonals
constexpr int SORT_RB = 4;                  // rim items of a thread in flight
constexpr long long SORT_WAIT_CYCLES = 4000000000LL;  // budget of a wait: about 2 s

// Words of SorTileArgs::sync.  The epoch (of the last half-sweep so far) goes
// on from launch to launch of a register tile's solver; the others are 0 at launch.
constexpr int SORT_SYNC_EPOCH = 0;
constexpr int SORT_SYNC_COUNT = 1;    // CTAs that have come to a grid barrier
constexpr int SORT_SYNC_LATE = 2;     // a CTA has given up a wait

// How a solve ends and where its checks come.
struct SorTileRun {
    int fixed;        // 1: exactly n iterations (max_iter), no test
    int n;            // fixed: iterations
    double tol;
    double tol2_above;  // a bound above tol^2: a larger ratio of the square sums is not converged
    int max_iter;
    int m;            // check interval
    int chunk;        // predicted checks: iterations are counted in chunks (0: check every m)
    const double *s_in;   // fixed: stored stencil of p_hi for the first residual if *s_ok (NULL: form it)
    double *s_out;        // fixed: where the final residual stores the stencil (NULL: nowhere)
    int *s_ok;            // fixed: 1 if the stencil is that of p_hi; 0 after a solve that gave up a wait
    long long wait;       // clock budget of a wait for another CTA (filled in by launch_tiles)
};

struct SorTileArgs {
    PDims d;
    SorTilePlan plan;
    float omega, h2;
    SorDiag dg;
    const float *b;
    double *p_hi;
    float *e[2], *r[2];
    double *partials;     // 2 per CTA
    uint4 *rim;           // published rim rows: [colour][tile][half][rim row][group]
    int rim_rows;         // rim rows of the largest tile
    unsigned *sync;       // SORT_SYNC_* words, then from word 32 a flag per tile, 32 words apart
    PoissonCtl *ctl;
};

// A rim row of a tile: its first group in the tile's arrays; the offset of
// its first group in a global colour array (r, and e as published), and
// those of its neighbours in y and z in other tiles (-1: none); bits of w:
// 0: colour parity for colour 0; 1: on the ground or lid plane; 2, 3: the
// row below / above in y is in the tile; 4, 5: in z; 6 .. 9: see sort_sweeps.
struct SorRimRow {
    int idx, roff, fy, fz;
    unsigned w;
};

// Dynamic shared memory of a tile of ty x tz rows: e (and r) of both
// colours, then the rim rows; of a register tile: e with its halo, r and
// the diagonals.
// With psm also the FP64 pressure of a register tile with its halo, and b.
inline size_t sort_smem_bytes(int nx, int ty, int tz, int G, bool rsmem, bool regs, bool psm)
{
    const size_t rows = (size_t)ty * tz;
    const size_t fixed = SORT_TILE_BYTES + SORT_KINDS * 32;
    const size_t padded = (size_t)(ty + 2) * (tz + 2);
    if (regs) return fixed + (padded + rows) * G * 32 + (psm ? (padded * 8 + rows * 4) * nx : 0);
    return fixed + rows * G * 32 * (rsmem ? 2 : 1) + (size_t)(2 * (ty + tz)) * sizeof(SorRimRow);
}

// A CTA's tile, at the start of its dynamic shared memory.  The phases of
// the solve are separate functions that read it (and keep their registers
// to themselves).
struct SorTile {
    SorTileArgs A;
    int G, threads;
    unsigned magic_g, magic_nx, magic_ty, magic_slots;  // of divisions by G, nx, ty and the slots of a row
    int ta, tb, py, ntiles;  // place of the tile
    int j0, k0, k1;          // first row, first and last plane
    int ty, tz, nrow;        // rows in y, planes, rows of the tile
    int ncol, ps, e0;        // groups of one colour of e, its plane step, its group 0 of row (0, 0)
    int nrim, rim_half;      // rim rows; 16-byte words of one half of a published rim
    unsigned barriers, epoch;  // grid barriers passed; epoch of the last half-sweep so far
    long long wait;          // clock budget of a wait for another CTA
    bool stored;             // the stored stencil is that of p_hi
    PoissonCtl c;
    double red[32];
};
static_assert(sizeof(SorTile) <= SORT_TILE_BYTES, "the tile's header");

extern __shared__ float4 sort_smem[];

__device__ __forceinline__ SorTile &sort_tile() { return *reinterpret_cast<SorTile *>(sort_smem); }

// e of a colour, r of a colour (where r is in shared memory), and what lies behind them
__device__ __forceinline__ float4 *sort_e(const SorTile &T, int colour) { return sort_smem + SORT_TILE_BYTES / 16 + colour * T.ncol; }
__device__ __forceinline__ float4 *sort_r(const SorTile &T, int colour)
{
    return sort_smem + SORT_TILE_BYTES / 16 + 2 * T.ncol + colour * T.nrow * T.G;
}

__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_gpu(unsigned *p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// A published word: two 64-bit elements {value, epoch}, each read and
// written whole.
__device__ __forceinline__ uint4 ld_relaxed_2x64(const uint4 *p)
{
    unsigned long long lo, hi;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}

__device__ __forceinline__ void st_relaxed_2x64(uint4 *p, float a, float b, unsigned epoch)
{
    const unsigned long long e = (unsigned long long)epoch << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(e | __float_as_uint(a)),
                 "l"(e | __float_as_uint(b)) : "memory");
}

// t / n for t n < 2^32 by a multiplication: magic = ceil(2^32 / n), 0 for n = 1.
__host__ __device__ inline unsigned sort_magic(unsigned n)
{
    return n > 1 ? (unsigned)(((1ull << 32) + n - 1) / n) : 0u;
}
__device__ __forceinline__ int sort_div(unsigned magic, unsigned t) { return magic ? (int)__umulhi(t, magic) : (int)t; }

// Row t of a tile's rim rows: jl | kl << 16 (the inverse of sort_rim_index).
__device__ __forceinline__ int sort_row_of(int t, int ty, int tz)
{
    if (t < ty) return t;
    if (t < 2 * ty) return (t - ty) | ((tz - 1) << 16);
    const int side = ty > 1 ? 2 : 1, n = t - 2 * ty;
    return (n % side ? ty - 1 : 0) | ((1 + n / side) << 16);
}

// Waits until *p has reached `target` (the count only grows); false after the clock budget.
__device__ __forceinline__ bool wait_reached(const unsigned *p, unsigned target, long long budget)
{
    const long long t0 = clock64();
    while ((int)(ld_relaxed_gpu(p) - target) < 0)
        if (clock64() - t0 > budget) return false;
    return true;
}

// Index of row (jl, kl) of a ty x tz tile among its rim rows: the first
// plane, the last plane, then the first and last row of the planes between.
__device__ __forceinline__ int sort_rim_index(int jl, int kl, int ty, int tz)
{
    if (kl == 0) return jl;
    if (kl == tz - 1) return ty + jl;
    const int side = ty > 1 ? 2 : 1;
    return 2 * ty + (kl - 1) * side + (jl == 0 ? 0 : side - 1);
}

// Two FP32 values in one 64-bit register, operated on together: one issue
// slot for two roundings, each the same as the scalar operation's.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pk(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float2 upk(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The diagonals of a group's four cells: -d and RN(1/d) (0, 0 past the row's end, which makes the update 0).
struct SorTileDiag {
    f32x2 nd[2], y[2];
};

// Two SOR updates: a, the x neighbours; ym .. zp, the others.  The division
// is sor_div's but for the sign of a zero quotient, which no later value
// depends on (the remainder's correction of an exact quotient adds 0).
__device__ __forceinline__ f32x2 sort_update2(f32x2 xl, f32x2 xr, f32x2 ym, f32x2 yp, f32x2 zm, f32x2 zp, f32x2 e,
                                              f32x2 r, f32x2 omega, f32x2 nh2, f32x2 nd, f32x2 y)
{
    const f32x2 s = add2(add2(add2(xl, xr), add2(ym, yp)), add2(zm, zp));
    const f32x2 x = fma2(nh2, r, s);
    const f32x2 q = mul2(x, y);
    const f32x2 gs = fma2(fma2(q, nd, x), y, q);
    return fma2(omega, fma2(e, pk(-1.0f, -1.0f), gs), e);
}

// Four SOR updates of one group.  q: colour parity of the row (x neighbours
// of slot s are slots s - 1 + q and s + q of the other colour); xe: the
// fifth x neighbour.
__device__ __forceinline__ float4 sort_update(const float4 &oc, float xe, bool q, const float4 &ym, const float4 &yp,
                                              const float4 &zm, const float4 &zp, const float4 &e, const float4 &r,
                                              f32x2 omega, f32x2 nh2, const SorTileDiag &D)
{
    const f32x2 a01 = pk(q ? oc.y : xe, q ? oc.z : oc.x), a23 = pk(q ? oc.w : oc.y, q ? xe : oc.z);
    const float2 u01 = upk(sort_update2(a01, pk(oc.x, oc.y), pk(ym.x, ym.y), pk(yp.x, yp.y), pk(zm.x, zm.y),
                                        pk(zp.x, zp.y), pk(e.x, e.y), pk(r.x, r.y), omega, nh2, D.nd[0], D.y[0]));
    const float2 u23 = upk(sort_update2(a23, pk(oc.z, oc.w), pk(ym.z, ym.w), pk(yp.z, yp.w), pk(zm.z, zm.w),
                                        pk(zp.z, zp.w), pk(e.z, e.w), pk(r.z, r.w), omega, nh2, D.nd[1], D.y[1]));
    return make_float4(u01.x, u01.y, u23.x, u23.y);
}

// Diagonals of the cells of group g in a row of parity q; lo: the row lies on the ground or lid plane.
__device__ __forceinline__ SorTileDiag sort_diag(const SorDiag &dg, int nx, int G, int g, bool q, bool lo)
{
    const float dm = lo ? 5.0f : 6.0f, ym = lo ? dg.y[1] : dg.y[2];
    float d[4] = {dm, dm, dm, dm}, y[4] = {ym, ym, ym, ym};
    if (g == 0 && !q) {  // i = 1
        d[0] = lo ? 4.0f : 5.0f;
        y[0] = lo ? dg.y[0] : dg.y[1];
    }
    if (g == G - 1) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = 2 * (4 * g + t) + 1 + q;
            if (i == nx) {
                d[t] = lo ? 6.0f : 7.0f;
                y[t] = lo ? dg.y[2] : dg.y[3];
            }
            if (i > nx) d[t] = y[t] = 0.0f;
        }
    }
    SorTileDiag D;
    D.nd[0] = pk(-d[0], -d[1]);
    D.nd[1] = pk(-d[2], -d[3]);
    D.y[0] = pk(y[0], y[1]);
    D.y[1] = pk(y[2], y[3]);
    return D;
}

#define SORT_OKP(idx) GBSW_INBOUNDS((long long)(idx), (long long)d.plane * (d.nz + 2), &g_sor_bounds)
#define SORT_OK4(idx) GBSW_INBOUNDS((long long)(idx), (long long)d.cplane * (d.nz + 2) - 3, &g_sor_bounds)

// Behind e and r: the diagonals by kind of group, then (I = 0) the rim rows.
__device__ __forceinline__ SorTileDiag *sort_diags(const SorTile &T, bool rsmem)
{
    return reinterpret_cast<SorTileDiag *>(sort_r(T, rsmem ? 2 : 0));
}

// Sum over the CTA in a fixed order; valid in thread 0.
__device__ __forceinline__ double sort_block_sum(double v, double *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = lane < nw ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    return v;
}

// Grid barrier; false (in every thread) if a wait gave up.
__device__ __noinline__ bool sort_grid_barrier()
{
    SorTile &T = sort_tile();
    __syncthreads();
    if (gridDim.x == 1) return true;
    bool late = false;
    if (threadIdx.x == 0) {
        const unsigned n = ++T.barriers;
        fence_gpu();
        atomicAdd(T.A.sync + SORT_SYNC_COUNT, 1u);
        late = !wait_reached(T.A.sync + SORT_SYNC_COUNT, n * gridDim.x, T.wait);
        fence_gpu();
    }
    return !__syncthreads_or(late);
}

// First published word of a rim row's neighbour in another tile, relative
// to its colour's first word; side 0, 1: below, above in y; 2, 3: in z.
__device__ __forceinline__ int sort_far_word(const SorTile &T, int side, int jl, int kl)
{
    const PDims &d = T.A.d;
    int tile, row;
    if (side < 2) {
        const int tn = side == 0 ? (T.ta > 0 ? T.ta - 1 : T.py - 1) : (T.ta < T.py - 1 ? T.ta + 1 : 0);
        const int tyn = (int)((long long)(tn + 1) * d.ny / T.py) - (int)((long long)tn * d.ny / T.py);
        tile = T.tb * T.py + tn;
        row = sort_rim_index(side == 0 ? tyn - 1 : 0, kl, tyn, T.tz);
    } else if (side == 2) {
        const int tzn = T.k0 - 1 - (int)((long long)(T.tb - 1) * d.nz / T.A.plan.pz);
        tile = T.tb * T.py + T.ta - T.py;
        row = sort_rim_index(jl, tzn - 1, T.ty, tzn);
    } else {
        tile = T.tb * T.py + T.ta + T.py;
        row = jl;
    }
    return tile * 2 * T.rim_half + row * T.G;
}

// A published group of a neighbouring tile.
struct SorFar {
    int o;  // its word, -1: no such neighbour
    uint4 a, b;
};

__device__ __forceinline__ void sort_far_load(const uint4 *from, int half, SorFar &f)
{
    if (f.o >= 0) {
        f.a = ld_relaxed_2x64(from + f.o);
        f.b = ld_relaxed_2x64(from + f.o + half);
    }
}

// Its values, once it carries the epoch (of the last half-sweep); *late if that does not come.
__device__ __forceinline__ float4 sort_far_get(const uint4 *from, int half, unsigned epoch, SorFar &f, long long budget,
                                               bool *late)
{
    if (f.o < 0) return make_float4(0.f, 0.f, 0.f, 0.f);
    if (f.a.y != epoch || f.a.w != epoch || f.b.y != epoch || f.b.w != epoch) {
        const long long t0 = clock64();
        do {
            if (clock64() - t0 > budget) {
                *late = true;
                break;
            }
            sort_far_load(from, half, f);
        } while (f.a.y != epoch || f.a.w != epoch || f.b.y != epoch || f.b.w != epoch);
    }
    return make_float4(__uint_as_float(f.a.x), __uint_as_float(f.a.z), __uint_as_float(f.b.x), __uint_as_float(f.b.z));
}

// Of a register tile (psm): the FP64 pressure with its halo and the right-hand side, in shared memory.
__device__ __forceinline__ double *sort_p(const SorTile &T)
{
    return reinterpret_cast<double *>(sort_diags(T, true) + SORT_KINDS);
}
__device__ __forceinline__ float *sort_b(const SorTile &T)
{
    return reinterpret_cast<float *>(sort_p(T) + (T.ty + 2) * (T.tz + 2) * T.A.d.nx);
}

// r = b - A p_hi in FP64 on the tile (as poisson_resid_kernel, bitwise), and
// the partial sums of r^2 and, with with_bb, of b^2.  s_in: the stencil is
// read, s_out: it is stored (FP64, padded layout).  p and b are in shared
// memory but for the halo; a thread takes single cells (dense over the tile:
// the FP64 pipe is the bound, and half-empty warps cost it as much as full
// ones), two at a time.
__device__ __noinline__ void sort_residual(const double *s_in, double *s_out, bool with_bb)
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int j0 = T.j0, k0 = T.k0, ty = T.ty, tz = T.tz, G = T.G, nx = d.nx;
    const double *p_hi = T.A.p_hi;
    const double r2 = d.rdx2;
    double rr = 0.0, bb = 0.0;
    if (!s_in && T.ntiles > 1) {
        // the halo: rows of the neighbouring tiles (or this one's own other side), 0 outside the grid in z
        double *P = sort_p(T);
        const int n = 2 * (ty + tz) * nx;
        for (int t0 = threadIdx.x; t0 < n; t0 += 4 * blockDim.x) {
            double v[4];
            int at[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int t = t0 + m * blockDim.x;
                at[m] = -1;
                if (t < n) {
                    const int row = sort_div(T.magic_nx, t), i = t - row * nx;
                    int jl, kl;
                    if (row < 2 * tz) {
                        jl = row < tz ? -1 : ty;
                        kl = row < tz ? row : row - tz;
                    } else {
                        kl = row < 2 * tz + ty ? -1 : tz;
                        jl = row - 2 * tz - (kl < 0 ? 0 : ty);
                    }
                    const int k = k0 + kl;
                    int j = j0 + jl;
                    j = j < 1 ? d.ny : (j > d.ny ? 1 : j);
                    const long long c = (long long)k * d.plane + (long long)j * d.pitch + i + 1;
                    at[m] = ((kl + 1) * (ty + 2) + jl + 1) * nx + i;
                    v[m] = k >= 1 && k <= d.nz && SORT_OKP(c) ? __ldcg(p_hi + c) : 0.0;
                }
            }
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (at[m] >= 0) P[at[m]] = v[m];
        }
        __syncthreads();
    }
    const int dk = (ty + 2) * nx, n = T.nrow * nx;
    const double *P = sort_p(T);
    const float *B = sort_b(T);
    float *const R0 = reinterpret_cast<float *>(sort_r(T, 0));
    const int other = 4 * T.nrow * G;
    for (int t0 = threadIdx.x; t0 < n; t0 += 2 * blockDim.x) {
        double res[2], bc[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int t = t0 + m * blockDim.x;
            res[m] = bc[m] = 0.0;
            if (t < n) {
                const int row = sort_div(T.magic_nx, t), i = t - row * nx + 1, kl = sort_div(T.magic_ty, row);
                const int jl = row - kl * ty, k = k0 + kl;
                double s;
                const long long c = (long long)k * d.plane + (long long)(j0 + jl) * d.pitch + i;
                if (s_in) {
                    s = SORT_OKP(c) ? s_in[c] : 0.0;
                } else {
                    const double *q = P + ((kl + 1) * (ty + 2) + jl + 1) * nx + i - 1;
                    // one tile: the rows below the first and above the last are its own other side
                    const int down = T.ntiles == 1 && jl == 0 ? (ty - 1) * nx : -nx;
                    const int up = T.ntiles == 1 && jl == ty - 1 ? -(ty - 1) * nx : nx;
                    const double w = i > 1 ? q[-1] : 0.0, e = i < nx ? q[1] : 0.0;
                    const double nb = (w + e) + (q[down] + q[up]) + (q[-dk] + q[dk]);
                    const int dci = 6 - (i == 1) - (k == 1) - (k == d.nz) + (i == nx);
                    const double dc = dci == 6 ? 6.0 : (dci == 5 ? 5.0 : (dci == 7 ? 7.0 : 4.0));
                    s = fma(-dc, q[0], nb);
                    if (s_out && SORT_OKP(c)) s_out[c] = s;
                }
                bc[m] = f64_from_f32(B[t]);
                res[m] = fma(-s, r2, bc[m]);
                R0[(((i + j0 + jl + k) & 1) ? other : 0) + 4 * row * G + ((i - 1) >> 1)] = f32_from_f64(res[m]);
            }
        }
        rr = fma(res[0], res[0], rr);
        rr = fma(res[1], res[1], rr);
        if (with_bb) {
            bb = fma(bc[0], bc[0], bb);
            bb = fma(bc[1], bc[1], bb);
        }
    }
    rr = sort_block_sum(rr, T.red);
    if (with_bb) bb = sort_block_sum(bb, T.red);
    if (threadIdx.x == 0) {
        T.A.partials[2 * blockIdx.x] = rr;
        if (with_bb) T.A.partials[2 * blockIdx.x + 1] = bb;
    }
}

// r of the tile into shared memory (a solve whose checks are kernels of their own).
__device__ __noinline__ void sort_read_r()
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int G = T.G, n = T.nrow * G, ty = T.ty;
    for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) {
        const int colour = t >= n, u = t - colour * n;
        const int row = sort_div(T.magic_g, u), g = u - row * G, kl = sort_div(T.magic_ty, row), jl = row - kl * ty;
        const long long c = (long long)(T.k0 + kl) * d.cplane + (long long)(T.j0 + jl) * d.cpitch + SOR_SLOT0 + 4 * g;
        sort_r(T, colour)[u] = SORT_OK4(c) ? __ldcg(reinterpret_cast<const float4 *>(T.A.r[colour] + c))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// With psm, before the first residual: the tile's copies of p and b.
__device__ __noinline__ void sort_read_tile()
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int nx = d.nx, ty = T.ty;
    double *P = sort_p(T);
    float *B = sort_b(T);
    for (int t = threadIdx.x; t < (ty + 2) * (T.tz + 2) * nx; t += blockDim.x) P[t] = 0.0;
    __syncthreads();
    for (int t = threadIdx.x; t < T.nrow * nx; t += blockDim.x) {
        const int row = sort_div(T.magic_nx, t), i = t - row * nx, kl = sort_div(T.magic_ty, row), jl = row - kl * ty;
        const long long c = (long long)(T.k0 + kl) * d.plane + (long long)(T.j0 + jl) * d.pitch + i + 1;
        P[((kl + 1) * (ty + 2) + jl + 1) * nx + i] = SORT_OKP(c) ? T.A.p_hi[c] : 0.0;
        B[t] = SORT_OKP(c) ? T.A.b[c] : 0.0f;
    }
    __syncthreads();
}

// e = 0 on the tile.
__device__ __forceinline__ void sort_clear_e(const SorTile &T)
{
    __syncthreads();
    float4 *E = sort_e(T, 0);
    for (int t = threadIdx.x; t < 2 * T.ncol; t += blockDim.x) E[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
}

// p_hi += e on the tile, e = 0; four slots (two cells each) in flight.
__device__ __noinline__ void sort_fold()
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int nx = d.nx, slots = (nx + 1) >> 1, ty = T.ty, G = T.G, ps = T.ps, e0 = T.e0, n = T.nrow * slots;
    double *p_hi = T.A.p_hi;
    const float *E0 = reinterpret_cast<const float *>(sort_e(T, 0));
    const int other = 4 * T.ncol;
    for (int t0 = threadIdx.x; t0 < n; t0 += 4 * blockDim.x) {
        double pa[4], pb[4];
        int at[4];  // element of p_hi (a grid that fits has fewer than 2^31)
        float ea[4], eb[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int t = t0 + m * blockDim.x;
            at[m] = -1;
            if (t < n) {
                const int row = sort_div(T.magic_slots, t), s = t - row * slots;
                const int kl = sort_div(T.magic_ty, row), jl = row - kl * ty, i = 2 * s + 1;
                const int c = (int)((long long)(T.k0 + kl) * d.plane) + (T.j0 + jl) * d.pitch + i;
                // cell i is of colour (i + j + k) & 1, cell i + 1 of the other (past the row's end: a pad slot, 0)
                const int c0 = (i + T.j0 + jl + T.k0 + kl) & 1;
                const int at_e = 4 * (e0 + kl * ps + jl * G) + s;
                ea[m] = E0[at_e + (c0 ? other : 0)];
                eb[m] = E0[at_e + (c0 ? 0 : other)];
                pa[m] = SORT_OKP(c) ? p_hi[c] : 0.0;
                pb[m] = SORT_OKP(c + 1) ? p_hi[c + 1] : 0.0;  // the ghost column at most
                at[m] = c;
            }
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (at[m] < 0) continue;
            if (SORT_OKP(at[m])) p_hi[at[m]] = pa[m] + f64_from_f32(ea[m]);
            if (eb[m] != 0.0f && SORT_OKP(at[m] + 1)) p_hi[at[m] + 1] = pb[m] + f64_from_f32(eb[m]);
        }
    }
    sort_clear_e(T);
}

// The same for a register tile with its own copy of p: the rows on the rim
// go to p_hi, where the neighbouring tiles read them, the others at the end.
__device__ __noinline__ void sort_fold_copy()
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int nx = d.nx, ty = T.ty, tz = T.tz, G = T.G, ps = T.ps, e0 = T.e0;
    double *P = sort_p(T);
    const float *E0 = reinterpret_cast<const float *>(sort_e(T, 0));
    const int other = 4 * T.ncol;
    for (int t = threadIdx.x; t < T.nrow * nx; t += blockDim.x) {
        const int row = sort_div(T.magic_nx, t), i = t - row * nx + 1, kl = sort_div(T.magic_ty, row), jl = row - kl * ty;
        const int c1 = (i + T.j0 + jl + T.k0 + kl) & 1;
        const float e = E0[4 * (e0 + kl * ps + jl * G) + ((i - 1) >> 1) + (c1 ? other : 0)];
        double *q = P + ((kl + 1) * (ty + 2) + jl + 1) * nx + i - 1;
        const double p = *q + f64_from_f32(e);
        *q = p;
        const long long c = (long long)(T.k0 + kl) * d.plane + (long long)(T.j0 + jl) * d.pitch + i;
        if ((jl == 0 || jl == ty - 1 || kl == 0 || kl == tz - 1) && SORT_OKP(c)) T.A.p_hi[c] = p;
    }
    sort_clear_e(T);
}

// The end of such a solve: the tile's p to p_hi.
__device__ __noinline__ void sort_write_tile()
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int nx = d.nx, ty = T.ty;
    for (int t = threadIdx.x; t < T.nrow * nx; t += blockDim.x) {
        const int row = sort_div(T.magic_nx, t), i = t - row * nx, kl = sort_div(T.magic_ty, row), jl = row - kl * ty;
        const long long c = (long long)(T.k0 + kl) * d.plane + (long long)(T.j0 + jl) * d.pitch + i + 1;
        if (SORT_OKP(c)) T.A.p_hi[c] = sort_p(T)[((kl + 1) * (ty + 2) + jl + 1) * nx + i];
    }
}

// n_iter iterations of a tile of any size.  A half-sweep updates the rim
// first (any row, its neighbours from shared memory or from the
// neighbouring tiles' published rows), then the rows inside it: what a
// neighbour reads was published a whole half-sweep of inner rows earlier.
// On the first half-sweep after a check every correction is 0 and no other
// tile is read.
template <bool RSMEM>
__device__ __noinline__ bool sort_sweeps(int n_iter)
{
    SorTile &T = sort_tile();
    const PDims &d = T.A.d;
    const int G = T.G, ty = T.ty, tz = T.tz, ps = T.ps, cpl = (int)d.cplane, cpitch = d.cpitch;
    const int nthreads = T.threads, tid = threadIdx.x, lane = tid & 31;
    const f32x2 om2 = pk(T.A.omega, T.A.omega), nh2 = pk(-T.A.h2, -T.A.h2);
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const SorTileDiag *diags = sort_diags(T, RSMEM);
    const SorRimRow *rim = reinterpret_cast<const SorRimRow *>(diags + SORT_KINDS);
    bool late = false;  // a wait of this thread gave up

    // ---- the inner march: unit u + lane is (z segment, row pair, group)
    const int nj = ty - 2, nk = tz - 2;  // inner rows and planes
    const int njb = nj > 0 ? (nj + 1) / 2 : 0;
    const int lseg = nk > 0 ? (nk + T.A.plan.nseg - 1) / T.A.plan.nseg : 0;
    const int nunits = (nj > 0 && nk > 0) ? njb * G * T.A.plan.nseg : 0;
    const int u0 = tid - lane;  // warp-uniform: the shuffles need whole warps
    const bool once = nunits <= nthreads;
    // place: first group, r of it in a global colour array, planes not stored
    // at the start, bits: 0, 1: first, last group of the row; 2: parity of
    // row jl at the first plane for colour 0; 3: the second row is inner too
    int base0 = 0, ro0 = 0, skip = 0;
    unsigned bits = 0;
    auto unit_at = [&](int u) {
        const int unit = min(u + lane, nunits - 1);
        const int cb = sort_div(T.magic_g, unit), g = unit - cb * G;
        const int seg = cb / njb, jl = 1 + 2 * (cb - seg * njb);
        // a segment is lseg planes long; the last one starts early enough to
        // end inside the tile and stores only its own planes
        const int k_own = 1 + seg * lseg, ks = min(k_own, tz - 1 - lseg);
        skip = u + lane < nunits ? k_own - ks : lseg;
        base0 = (ks * ty + jl) * G + g;
        bits = (g == 0) | ((g == G - 1) << 1) | (((1 + T.j0 + jl + T.k0 + ks) & 1) << 2) | ((jl + 1 <= ty - 2) << 3);
        ro0 = (int)((long long)(T.k0 + ks) * d.cplane + (long long)(T.j0 + jl) * cpitch + SOR_SLOT0 + 4 * g);
    };
    auto load_r = [&](const float *rg, int o) -> float4 {
        return SORT_OK4(o) ? __ldcg(reinterpret_cast<const float4 *>(rg + o)) : zero4;
    };
    float4 ra[2], rb[2];
    auto first_r = [&](const float *rg) {  // r of the first two planes (the arrays have a plane past the last one)
        ra[0] = load_r(rg, ro0);
        rb[0] = load_r(rg, ro0 + cpitch);
        ra[1] = load_r(rg, ro0 + cpl);
        rb[1] = load_r(rg, ro0 + cpl + cpitch);
    };
    if (u0 < nunits) unit_at(u0);

    // r of a thread's first rim items, read before the barrier that precedes them
    float4 r4[SORT_RB];
    auto rim_r = [&](const float *rg, int t0) {
#pragma unroll
        for (int n = 0; n < SORT_RB; ++n) {
            const int t = t0 + n * nthreads;
            if (t < T.nrim * G) {
                const int row = sort_div(T.magic_g, t);
                r4[n] = load_r(rg, rim[row].roff + 4 * (t - row * G));
            }
        }
    };
    if (!RSMEM) rim_r(T.A.r[0], tid);
    // the flag of a neighbouring tile that this lane watches for its warp
    int nb = -1;
    if (lane == 0 && T.py > 1) nb = T.tb * T.py + (T.ta + T.py - 1) % T.py;
    if (lane == 1 && T.py > 1) nb = T.tb * T.py + (T.ta + 1) % T.py;
    if (lane == 2 && T.tb > 0) nb = (int)blockIdx.x - T.py;
    if (lane == 3 && T.k1 < d.nz) nb = (int)blockIdx.x + T.py;
    const unsigned *flag = T.A.sync + 32 * (1 + max(nb, 0));
    // the other tiles' rows beside a thread's first rim items (the row beside
    // a corner row in y is read when its turn comes)
    float4 vf[SORT_RB];
    auto rim_far = [&](const float *eo, int t0, bool far) {
#pragma unroll
        for (int n = 0; n < SORT_RB; ++n) {
            const int t = t0 + n * nthreads;
            vf[n] = zero4;
            if (far && t < T.nrim * G) {
                const int row = sort_div(T.magic_g, t), g = t - row * G;
                const int fy = rim[row].fy, fz = rim[row].fz, f = fz >= 0 ? fz : fy;
                if (f >= 0) vf[n] = load_r(eo, f + 4 * g);
            }
        }
    };
    rim_far(nullptr, tid, false);

    for (int h = 0; h < 2 * n_iter; ++h) {
        const int colour = h & 1;
        const float4 *O = sort_e(T, 1 - colour);
        float4 *C = sort_e(T, colour);
        const float4 *RR = sort_r(T, colour);
        const float *rg = colour ? T.A.r[1] : T.A.r[0];
        {
            const int nitems = T.nrim * G;
            const bool far = h > 0;
            const float *eo = colour ? T.A.e[0] : T.A.e[1];
            float *ec = colour ? T.A.e[1] : T.A.e[0];
            int t0 = tid;
            asm volatile("" : "+r"(t0));  // the items' addresses are formed anew each time, not kept in registers
            for (; t0 < nitems; t0 += SORT_RB * nthreads) {
                if (t0 >= SORT_RB * nthreads) {  // the first items' reads were issued before
                    rim_far(eo, t0, far);
                    if (!RSMEM) rim_r(rg, t0);
                }
#pragma unroll
                for (int n = 0; n < SORT_RB; ++n) {
                    const int t = t0 + n * nthreads;
                    if (t < nitems) {
                        const int row = sort_div(T.magic_g, t), g = t - row * G;
                        const int idx = rim[row].idx + g, off = rim[row].roff + 4 * g;
                        const unsigned w = rim[row].w;
                        const int kind = ((w ^ (unsigned)colour) & 1u) << 2 | (w & 2u) << 2 | (g == 0) | (g == G - 1) << 1;
                        const bool q = kind & 4;
                        float xe = reinterpret_cast<const float *>(O + idx)[q ? 4 : -1];
                        float4 vy = vf[n];
                        if (rim[row].fy >= 0 && rim[row].fz >= 0) vy = far ? load_r(eo, rim[row].fy + 4 * g) : zero4;
                        const float4 vz = rim[row].fz >= 0 ? vf[n] : zero4;
                        float4 ym = vy, yp = vy, zm = vz, zp = vz;
                        if (w & 4u) ym = O[idx - G];
                        if (w & 8u) yp = O[idx + G];
                        if (w & 16u) zm = O[idx - ps];
                        if (w & 32u) zp = O[idx + ps];
                        if (w & 960u) {
                            // 64, 128: the row wraps to the tile's own other side; 256: the
                            // tile's only row, vy is the row below; 512: its only plane, vz
                            // is the row below if there is one, else the one above
                            if (w & 64u) ym = O[idx + (ty - 1) * G];
                            if (w & 128u) yp = O[idx - (ty - 1) * G];
                            if (w & 256u)
                                yp = far ? load_r(eo, off + (T.j0 == d.ny ? 1 - d.ny : 1) * cpitch) : zero4;
                            if (w & 512u) {
                                if (T.tb > 0) zp = far && T.k1 < d.nz ? load_r(eo, off + cpl) : zero4;
                                else zm = zero4;
                            }
                        }
                        if (kind & (q ? 2 : 1)) xe = 0.0f;
                        const float4 u = sort_update(O[idx], xe, q, ym, yp, zm, zp, C[idx], RSMEM ? RR[idx] : r4[n], om2,
                                                     nh2, diags[kind]);
                        C[idx] = u;
                        if (SORT_OK4(off)) __stcg(reinterpret_cast<float4 *>(ec + off), u);
                    }
                }
            }
            if (T.ntiles > 1) {  // this warp's rim rows are published
                __syncwarp();
                if (lane == 0) red_release_gpu(T.A.sync + 32 * (1 + blockIdx.x), 1u);
            }
        }
        // The neighbours' rim rows of this half-sweep, which the next one
        // reads: their flags are looked at in the middle of the march, by
        // when they are usually set, and the rows then read ahead.
        const unsigned target = (T.epoch + h + 1) * (unsigned)(nthreads >> 5);
        bool fetched = h + 1 == 2 * n_iter;  // no next half-sweep: nothing to read
        const float *next_far = colour ? T.A.e[1] : T.A.e[0];
        auto look = [&]() {
            const bool set = nb < 0 || (int)(ld_acquire_gpu(flag) - target) >= 0;
            if (__all_sync(0xffffffffu, set)) {
                __syncwarp();
                int t0 = tid;
                asm volatile("" : "+r"(t0));
                rim_far(next_far, t0, true);
                fetched = true;
            }
        };
        for (int u = u0; u < nunits; u += nthreads) {
            if (!once) unit_at(u);
            if (!RSMEM) first_r(rg);
            const bool two = bits & 8u, q0 = ((bits >> 2) ^ colour) & 1u;
            const int kA = (bits & 3u) | q0 << 2, kB = kA ^ 4;
            // diagonals of row jl on even and odd steps of the march (row jl + 1: the other one)
            const SorTileDiag DA = diags[kA], DB = diags[kB];
            int base = base0, ro = ro0 + 2 * cpl;
            const int op_off = two ? 2 * G : 0;
            // the neighbouring lane holds the adjacent group unless this is the row's end or the warp's
            const bool edge0 = lane == 0 && !(bits & 1u), edge1 = lane == 31 && !(bits & 2u);
            auto fifth = [&](const float4 &v, bool q, int b0) -> float {
                float x = __shfl_sync(0xffffffffu, q ? v.x : v.w, (lane + (q ? 1 : 31)) & 31);
                if (q ? edge1 : edge0) x = reinterpret_cast<const float *>(O + b0)[q ? 4 : -1];
                return bits & (q ? 2u : 1u) ? 0.0f : x;
            };
            // One plane of the two rows: p, c, n: the other colour's vectors of
            // the planes below, here and above; m, q: of the rows below and
            // above; e: the rows' own.  Those of the next plane are read right
            // after this one is updated (the plane above the next in place of
            // the plane below).
            float4 om = O[base - G], oq = O[base + op_off], ea = C[base], eb = C[base + G];
            auto step = [&](int n, float4 &pa, float4 &pb, const float4 &ca, const float4 &cb, const float4 &na,
                            const float4 &nb, float4 &r0, float4 &r1, bool q, const SorTileDiag &D0,
                            const SorTileDiag &D1) {
                const float xa = fifth(ca, q, base), xb = fifth(cb, !q, base + G);
                const float4 ua = sort_update(ca, xa, q, om, cb, pa, na, ea, RSMEM ? RR[base] : r0, om2, nh2, D0);
                const float4 ub = sort_update(cb, xb, !q, ca, oq, pb, nb, eb, RSMEM ? RR[base + G] : r1, om2, nh2, D1);
                if (n >= skip) {
                    C[base] = ua;
                    if (two) C[base + G] = ub;
                }
                if (n + 1 >= lseg) return;
                base += ps;
                om = O[base - G];
                oq = O[base + op_off];
                ea = C[base];
                eb = C[base + G];
                pa = O[base + ps];
                pb = O[base + ps + G];
                if (!RSMEM && n + 2 < lseg) {
                    r0 = load_r(rg, ro);
                    r1 = load_r(rg, ro + cpitch);
                    ro += cpl;
                }
            };
            float4 a0 = O[base - ps], b0 = O[base - ps + G], a1 = O[base], b1 = O[base + G];
            float4 a2 = O[base + ps], b2 = O[base + ps + G];
            for (int n = 0; n < lseg; n += 6) {
                step(n, a0, b0, a1, b1, a2, b2, ra[0], rb[0], q0, DA, DB);
                if (n + 1 >= lseg) break;
                step(n + 1, a1, b1, a2, b2, a0, b0, ra[1], rb[1], !q0, DB, DA);
                if (n + 2 >= lseg) break;
                if (!fetched && n == 0) look();
                step(n + 2, a2, b2, a0, b0, a1, b1, ra[0], rb[0], q0, DA, DB);
                if (n + 3 >= lseg) break;
                step(n + 3, a0, b0, a1, b1, a2, b2, ra[1], rb[1], !q0, DB, DA);
                if (n + 4 >= lseg) break;
                step(n + 4, a1, b1, a2, b2, a0, b0, ra[0], rb[0], q0, DA, DB);
                if (n + 5 >= lseg) break;
                step(n + 5, a2, b2, a0, b0, a1, b1, ra[1], rb[1], !q0, DB, DA);
            }
        }
        if (!fetched) {
            if (nb >= 0) late = !wait_reached(flag, target, T.wait);
            __syncwarp();
            look();
        }
        if (!RSMEM) {
            int t0 = tid;
            asm volatile("" : "+r"(t0));
            rim_r(colour ? T.A.r[0] : T.A.r[1], t0);
        }
        if (__syncthreads_or(late)) return false;
    }
    return true;
}

// n_iter iterations of a register tile: e has a halo of one row on every
// side, which the threads fill from the neighbouring tiles' published rows;
// then every thread updates its I groups, whose e (and r, for I <= 2) stay
// in its registers.  One barrier per half-sweep: a half-sweep fills the
// halo of one colour and writes the rows of the other.
template <int I>
__device__ __noinline__ bool sort_register_sweeps(int n_iter)
{
    constexpr bool RREG = I <= 2;  // else r is read from shared memory
    SorTile &T = sort_tile();
    const int G = T.G, ty = T.ty, tz = T.tz, ps = T.ps, e0 = T.e0, ngroups = T.nrow * G, half_words = T.rim_half;
    const int nthreads = T.threads, tid = threadIdx.x;
    const unsigned magic = T.magic_g;
    const bool many = T.ntiles > 1;
    const f32x2 om2 = pk(T.A.omega, T.A.omega), nh2 = pk(-T.A.h2, -T.A.h2);
    const SorTileDiag *diags = sort_diags(T, true);
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    unsigned epoch = T.epoch;
    bool late = false;  // a wait of this thread gave up
    float4 e[I][2], r[RREG ? I : 1][2];
    int idx[I], pub[I], kind[I], wrap[I];  // group in e, published word, diagonals of colour 0, copy in the halo
#pragma unroll
    for (int m = 0; m < I; ++m) {
        const int t = tid + m * nthreads, tc = min(t, ngroups - 1);
        const int row = sort_div(magic, tc), g = tc - row * G;
        const int kl = sort_div(T.magic_ty, row), jl = row - kl * ty, k = T.k0 + kl;
        idx[m] = t < ngroups ? e0 + kl * ps + jl * G + g : -1;
        pub[m] = many && (jl == 0 || jl == ty - 1 || kl == 0 || kl == tz - 1) ? sort_rim_index(jl, kl, ty, tz) * G + g : -1;
        wrap[m] = T.py > 1 ? 0 : (jl == 0 ? ty * G : (jl == ty - 1 ? -ty * G : 0));
        kind[m] = (g == 0) | ((g == G - 1) << 1) | (((1 + T.j0 + jl + k) & 1) << 2) | ((k == 1 || k == T.A.d.nz) << 3);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            e[m][q] = zero4;
            if (RREG) r[m][q] = t < ngroups ? sort_r(T, q)[t] : zero4;
        }
    }
    int hsrc[SORT_HALO], hdst[SORT_HALO];  // halo groups that this thread fetches
    const int nhalo = 2 * (ty + tz) * G;
#pragma unroll
    for (int m = 0; m < SORT_HALO; ++m) {
        const int t = tid + m * nthreads;
        hsrc[m] = -1;
        hdst[m] = 0;
        if (t < nhalo) {
            int row = sort_div(magic, t);
            const int g = t - row * G;
            if (row < 2 * tz) {
                const int s = row >= tz, kl = row - s * tz;
                if (T.py > 1) hsrc[m] = sort_far_word(T, s, 0, kl) + g;
                hdst[m] = e0 + kl * ps + (s ? ty : -1) * G + g;
            } else {
                row -= 2 * tz;
                const int s = row >= ty, jl = row - s * ty;
                if (s ? T.k1 < T.A.d.nz : T.k0 > 1) hsrc[m] = sort_far_word(T, 2 + s, jl, 0) + g;
                hdst[m] = e0 + (s ? tz : -1) * ps + jl * G + g;
            }
        }
    }
    auto half = [&](auto cc, bool halo) -> bool {
        constexpr int colour = decltype(cc)::value;
        float4 *O = sort_e(T, 1 - colour), *C = sort_e(T, colour);
        if (halo && many) {
            const uint4 *from = T.A.rim + (long long)(1 - colour) * T.ntiles * 2 * half_words;
#pragma unroll
            for (int m = 0; m < SORT_HALO; m += 2) {  // two in flight
                if (m * nthreads < nhalo) {
                    SorFar f0, f1;
                    f0.o = hsrc[m];
                    f1.o = hsrc[m + 1];
                    sort_far_load(from, half_words, f0);
                    sort_far_load(from, half_words, f1);
                    if (f0.o >= 0) O[hdst[m]] = sort_far_get(from, half_words, epoch, f0, T.wait, &late);
                    if (f1.o >= 0) O[hdst[m + 1]] = sort_far_get(from, half_words, epoch, f1, T.wait, &late);
                }
            }
        }
        if (__syncthreads_or(late)) return false;
        uint4 *mine = T.A.rim + ((long long)colour * T.ntiles + (int)blockIdx.x) * 2 * half_words;
        const float4 *RR = sort_r(T, colour);
#pragma unroll
        for (int m = 0; m < I; ++m) {
            const int c0 = idx[m];
            if (c0 >= 0) {
                const int kd = colour ? kind[m] ^ 4 : kind[m];
                const bool q = kd & 4;
                const float4 oc = O[c0];
                float xe = reinterpret_cast<const float *>(O + c0)[q ? 4 : -1];
                if (q ? kd & 2 : kd & 1) xe = 0.0f;
                const float4 u = sort_update(oc, xe, q, O[c0 - G], O[c0 + G], O[c0 - ps], O[c0 + ps], e[m][colour],
                                             RREG ? r[RREG ? m : 0][colour] : RR[tid + m * nthreads], om2, nh2, diags[kd]);
                e[m][colour] = u;
                if (pub[m] >= 0) {
                    st_relaxed_2x64(mine + pub[m], u.x, u.y, epoch + 1);
                    st_relaxed_2x64(mine + half_words + pub[m], u.z, u.w, epoch + 1);
                }
                C[c0] = u;
                if (wrap[m]) C[c0 + wrap[m]] = u;
            }
        }
        ++epoch;
        return true;
    };
    for (int it = 0; it < n_iter; ++it) {
        if (!half(std::integral_constant<int, 0>{}, it > 0)) return false;
        if (!half(std::integral_constant<int, 1>{}, true)) return false;
    }
    return true;
}

// Thread 0: the convergence test and the place of the next check (as
// poisson_test_kernel), on the residual's square sums.  The control block's
// `next` becomes the iterations until the next check, 0 when the solve is done.
__device__ __noinline__ void sort_test(const SorTileRun &run, bool counting, int ran, double rr, double bb)
{
    PoissonCtl &c = sort_tile().c;
    if (counting) {
        c.iters += ran;
    } else {
        c = PoissonCtl{};
        c.status = DEV_OK;
        c.bb = bb;
    }
    const double rr_prev = c.rr;  // of the check before, `ran` iterations ago
    c.rr = rr;
    // Far from the tolerance: no root, no logarithm, no division (a few us in
    // FP64).  A prediction then has no say if the tolerance is more than m
    // iterations away: tol / rho < rho / rho_prev over at least m iterations.
    if (counting && !run.fixed && (run.chunk == 0 || run.chunk >= run.m) && isfinite(rr) && c.bb >= 1e-60 &&
        rr > c.bb * run.tol2_above && c.iters < run.max_iter &&
        (run.chunk == 0 || rr * rr > run.tol2_above * rr_prev * c.bb * (1.0 + 1e-9))) {
        c.next = run.chunk > 0 ? run.chunk : run.m;
        return;
    }
    const double rho = c.bb > 0.0 ? sqrt(rr / c.bb) : 0.0;
    c.rho = rho;
    const bool bad = !isfinite(rr) || !isfinite(c.bb) || !isfinite(rho);
    if (bad) c.status = DEV_NONFINITE;
    const int most = run.fixed ? run.n : run.max_iter;
    const bool done = bad || c.bb < 1e-60 || rho <= run.tol || c.iters >= most;
    c.done = done ? 1 : 0;
    int next = run.m;
    const double rho_prev = c.bb > 0.0 ? sqrt(rr_prev / c.bb) : 0.0;
    if (run.chunk > 0 && counting && !done && rho > 0.0 && rho < rho_prev && ran > 0) {
        const double lg = log(rho / rho_prev) / (double)ran;
        const double n = log(run.tol / rho) / lg;
        if (n < (double)run.m) next = max(1, (int)ceil(1.03 * n) + 1);
    }
    next = max(1, min(next, run.max_iter - c.iters));
    if (run.fixed) c.next = counting ? 0 : run.n;
    else if (done) c.next = 0;
    else c.next = run.chunk > 0 ? run.chunk * ((next + run.chunk - 1) / run.chunk) : run.m;
}

// Cooperative launch: grid py * pz, block plan.threads.  I = 0: a tile of
// any size; I > 0: a tile of at most I * plan.threads
// groups, each thread keeping e (and r) of its I groups in registers.
template <int I, bool RSMEM>
__global__ void __launch_bounds__(I ? SORT_SMALL_THREADS : SORT_THREADS, 1)
sor_solve_kernel(const __grid_constant__ SorTileArgs A, const __grid_constant__ SorTileRun run)
{
    SorTile &T = sort_tile();
    const int tid = threadIdx.x;
    if (tid == 0) {
        const SorTilePlan &P = A.plan;
        T.A = A;
        T.G = P.G;
        T.threads = P.threads;
        T.magic_g = P.magic_g;
        T.magic_nx = sort_magic(A.d.nx);
        T.magic_slots = sort_magic((A.d.nx + 1) >> 1);
        T.py = P.py;
        T.ntiles = P.py * P.pz;
        T.ta = blockIdx.x % P.py;
        T.tb = blockIdx.x / P.py;
        T.j0 = (int)((long long)T.ta * A.d.ny / P.py) + 1;
        T.k0 = (int)((long long)T.tb * A.d.nz / P.pz) + 1;
        T.k1 = (int)((long long)(T.tb + 1) * A.d.nz / P.pz);
        T.ty = (int)((long long)(T.ta + 1) * A.d.ny / P.py) - T.j0 + 1;
        T.tz = T.k1 - T.k0 + 1;
        T.magic_ty = sort_magic(T.ty);
        T.nrow = T.ty * T.tz;
        // e of a register tile has a halo of one row on every side
        const int ety = I ? T.ty + 2 : T.ty;
        T.ncol = ety * (I ? T.tz + 2 : T.tz) * P.G;
        T.ps = ety * P.G;
        T.e0 = I ? T.ps + P.G : 0;
        T.nrim = T.tz > 2 ? 2 * T.ty + (T.ty > 1 ? 2 : 1) * (T.tz - 2) : T.nrow;
        T.rim_half = A.rim_rows * P.G;
        T.barriers = 0;
        T.wait = run.wait;
        T.stored = run.s_in && *run.s_ok != 0;
        T.epoch = A.sync[SORT_SYNC_EPOCH];
    }
    __syncthreads();
    SorTileDiag *diags = sort_diags(T, RSMEM);
    if (tid < SORT_KINDS)  // bits 0, 1: first, last group; 2: parity; 3: ground or lid plane
        diags[tid] = sort_diag(A.dg, A.d.nx, (tid & 2) ? T.G : T.G + 1, (tid & 1) ? 0 : T.G - 1, tid & 4, tid & 8);
    SorRimRow *rim = reinterpret_cast<SorRimRow *>(diags + SORT_KINDS);
    for (int t = tid; t < (I ? 0 : T.nrim); t += blockDim.x) {
        const int rk = sort_row_of(t, T.ty, T.tz), kl = rk >> 16, jl = rk & 0xffff;
        const int j = T.j0 + jl, k = T.k0 + kl, ty = T.ty, tz = T.tz;
        SorRimRow w;
        w.idx = (kl * ty + jl) * T.G;
        w.roff = (int)((long long)k * A.d.cplane + (long long)j * A.d.cpitch + SOR_SLOT0);
        w.fy = w.fz = -1;
        if (T.py > 1 && jl == 0) w.fy = w.roff + ((j == 1 ? A.d.ny : j - 1) - j) * A.d.cpitch;
        else if (T.py > 1 && jl == ty - 1) w.fy = w.roff + ((j == A.d.ny ? 1 : j + 1) - j) * A.d.cpitch;
        if (kl == 0 && k > 1) w.fz = w.roff - (int)A.d.cplane;
        else if (kl == tz - 1 && k < A.d.nz) w.fz = w.roff + (int)A.d.cplane;
        w.w = ((1 + j + k) & 1) | ((k == 1 || k == A.d.nz) ? 2u : 0u) | (jl > 0 ? 4u : 0u) | (jl < ty - 1 ? 8u : 0u) |
              (kl > 0 ? 16u : 0u) | (kl < tz - 1 ? 32u : 0u) | (T.py == 1 && jl == 0 ? 64u : 0u) |
              (T.py == 1 && jl == ty - 1 ? 128u : 0u) | (T.py > 1 && ty == 1 ? 256u : 0u) | (tz == 1 ? 512u : 0u);
        rim[t] = w;
    }
    {
        float4 *all = sort_e(T, 0);
        const int n = 2 * T.ncol + (RSMEM ? 2 : 0) * T.nrow * T.G;
        for (int t = tid; t < n; t += blockDim.x) all[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();

    // Checks as kernels of their own: run.n iterations, or with run.n < 0 those until the next check.
    if (!A.plan.psm) {
        int n = run.n;
        if (n < 0) n = run.chunk * ((A.ctl->next + run.chunk - 1) / run.chunk);
        if (RSMEM) sort_read_r();
        __syncthreads();
        bool ok;
        if constexpr (I > 0) ok = sort_register_sweeps<I>(n);
        else ok = sort_sweeps<RSMEM>(n);
        if (ok) {
            __syncthreads();
            sort_fold();
            if (I > 0) ok = sort_grid_barrier();  // every CTA has read the epoch
        }
        if (tid == 0) {
            if (!ok) {
                atomicCAS(&A.ctl->status, DEV_OK, DEV_TIMEOUT);
                if (atomicExch(A.sync + SORT_SYNC_LATE, 1u) == 0) atomicAdd(A.sync + SORT_SYNC_EPOCH, 1u << 24);
            } else if (blockIdx.x == 0) {
                A.ctl->since = n;
                if (I > 0) atomicAdd(A.sync + SORT_SYNC_EPOCH, 2u * n);
            }
        }
        return;
    }
    if constexpr (I > 0) {
        bool ok, first = true;
        int ran = 0;
        sort_read_tile();
        for (;;) {
            sort_residual(first && T.stored ? run.s_in : nullptr, !first && run.fixed ? run.s_out : nullptr, first);
            ok = sort_grid_barrier();
            if (!ok) break;
            if (tid < 32) {
                // the CTAs' partial sums in a fixed order, the same in every CTA
                double rr = 0.0, bb = 0.0;
                for (int q0 = tid; q0 < (int)gridDim.x; q0 += 5 * 32) {
                    double v[5];
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        const int q = q0 + 32 * m;
                        v[m] = q < (int)gridDim.x ? __ldcg(A.partials + 2 * q) : 0.0;
                    }
#pragma unroll
                    for (int m = 0; m < 5; ++m) rr += v[m];
                }
                if (first)
                    for (int q = tid; q < (int)gridDim.x; q += 32) bb += __ldcg(A.partials + 2 * q + 1);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    rr += __shfl_down_sync(0xffffffffu, rr, o);
                    if (first) bb += __shfl_down_sync(0xffffffffu, bb, o);
                }
                if (tid == 0) sort_test(run, !first, ran, rr, bb);
            }
            __syncthreads();
            ran = T.c.next;
            if (ran == 0 && !(run.fixed && first)) break;  // a fixed count of 0 still forms the final residual
            first = false;
            ok = sort_register_sweeps<I>(ran);
            if (!ok) break;
            __syncthreads();
            if (tid == 0) T.epoch += 2 * ran;
            sort_fold_copy();
            ok = sort_grid_barrier();
            if (!ok) break;
        }
        if (ok) sort_write_tile();
        if (tid == 0) {
            // One CTA may pass the last barrier while another gives it up, its
            // part of p not written: the solve has then failed, whichever of the
            // two comes here first.  The one raises the flag, then the status;
            // the other writes its status, then looks at the flag.  (s_ok too.)
            if (!ok) {
                const bool first_late = atomicExch(A.sync + SORT_SYNC_LATE, 1u) == 0;
                __threadfence();
                atomicExch(&A.ctl->status, DEV_TIMEOUT);
                if (run.s_out) atomicExch(run.s_ok, 0);
                // past every epoch that this solve may have published
                if (first_late) atomicAdd(A.sync + SORT_SYNC_EPOCH, 1u << 24);
            } else if (blockIdx.x == 0) {
                *A.ctl = T.c;
                A.sync[SORT_SYNC_EPOCH] = T.epoch;
                if (run.s_out) *run.s_ok = 1;
                __threadfence();
                if (ld_relaxed_gpu(A.sync + SORT_SYNC_LATE)) {
                    atomicExch(&A.ctl->status, DEV_TIMEOUT);
                    if (run.s_out) atomicExch(run.s_ok, 0);
                }
            }
        }
    }
}
#undef SORT_OKP
#undef SORT_OK4

}  // namespace gbsw
