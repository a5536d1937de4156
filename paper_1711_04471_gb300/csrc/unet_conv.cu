// tcgen05 implicit-GEMM 3x3x3 convolution (see unet_conv.cuh for the data
// layout and the pipeline), weight packing, and the operator-level C ABI
// used to check the kernel against the FP64 oracle.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "unet_conv.cuh"
#include "unet_internal.cuh"

namespace gbsw {

namespace {

constexpr int CONV_THREADS = 128;

__device__ __forceinline__ void set_status(int *status, int code) { atomicCAS(status, DEV_OK, code); }

// Where a tile lies: z0 = sample * D + z; planes: how many of its box_z planes exist.
struct TilePos {
    int x0, y0, z0, sample, z, planes;
};

__device__ __forceinline__ TilePos tile_pos(const ConvGeom &g, int t)
{
    TilePos p;
    p.x0 = (t % g.tiles_x) * g.box_x;
    t /= g.tiles_x;
    p.y0 = (t % g.tiles_y) * g.box_y;
    t /= g.tiles_y;
    if (g.sample_tiles == 0) {  // whole samples: the last tile may hold fewer
        p.z0 = t * g.box_z;
        p.sample = p.z0 / g.D;
        p.z = 0;
        p.planes = g.NZ - p.z0;
    } else {
        p.sample = t / g.sample_tiles;
        p.z = (t - p.sample * g.sample_tiles) * g.box_z;
        p.z0 = p.sample * g.D + p.z;
        p.planes = g.D - p.z;
    }
    return p;
}

// One thread: the tile at p shifted by (dx, dy, dz), one box with all channel
// groups into slabs of 2048 bytes at dst; the whole box arrives on bar, zeros
// where it lies outside the sample.
__device__ __forceinline__ void load_tile(uint8_t *dst, const CUtensorMap *map, uint64_t *bar, const ConvGeom &g,
                                          const TilePos &p, int dx, int dy, int dz)
{
    const int x = p.x0 + dx, y = p.y0 + dy, z = p.z + dz;
    if (g.load == LOAD_SAMPLES) {
        tc::tma_load_5d(dst, map, bar, 8 * x, y, z, p.sample, 0);
        return;
    }
    const int zsrc = z >= 0 && z < g.D ? p.z0 + dz : -1;
    if (g.load == LOAD_ROWS) tc::tma_load_5d(dst, map, bar, 8 * x, y, 0, zsrc, 0);
    else tc::tma_load_5d(dst, map, bar, 0, x, y, 0, zsrc);
}

template <int CIN, int COUT>
struct ConvSmem {
    static constexpr int A_BYTES = 128 * CIN * 2;
    static constexpr int B_BYTES = COUT * CIN * 2;
    static constexpr int STAGE = ((A_BYTES + B_BYTES + 1023) / 1024) * 1024;
    // Taps in flight.  Four leave room for more tiles per SM, whose epilogues
    // overlap; with few tiles only the ring hides the loads' latency, of which
    // little is left (16 -> 16 channels: 8192 tiles 75 us with 4, 111 with 9;
    // 32 -> 64, 8 tiles 13.0 with 4, 12.7 with 6).  64 input channels leave room
    // for four only.
    static constexpr int STAGES = 4;
    static constexpr int FIT = 72 * 1024 / STAGE;  // what leaves room for a weight-gradient CTA on the SM
    static constexpr int DEEP = FIT > 9 ? 9 : FIT < STAGES ? STAGES : FIT;
    static constexpr int bytes(int stages) { return stages * STAGE + 256 + 1024; }  // barriers + TMEM slot, alignment slack
    static constexpr int TMEM_COLS = COUT < 32 ? 32 : COUT;
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(CONV_THREADS)
conv3d_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __nv_bfloat16 *__restrict__ wpack,
                 const float *__restrict__ bias, __nv_bfloat16 *__restrict__ y, float *__restrict__ y_f32,
                 const __nv_bfloat16 *__restrict__ mask, ConvGeom g, int epi, int stages, int *status)
{
    using S = ConvSmem<CIN, COUT>;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 256, "UMMA shape");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + stages * S::STAGE);
    uint64_t *empty = full + stages;
    uint64_t *done = empty + stages;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const TilePos pos = tile_pos(g, blockIdx.x);
    // the taps of a single-plane tile that stay in the sample: a range
    const bool multi = g.box_z > 1;  // tile of several planes (small planes)
    const int tap_begin = !multi && pos.z == 0 ? 9 : 0, tap_end = !multi && pos.z == g.D - 1 ? 18 : 27;

    if (warp == 0) {
        tc::tmem_alloc(tmem_slot, S::TMEM_COLS);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < stages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(done, 1);
        tc::fence_mbar_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (threadIdx.x == 0) {
        // producer: one stage per tap
        int dx = -1, dy = -1, dz = tap_begin / 9 - 1, s = 0, parity = 1;
        for (int tap = tap_begin; tap < tap_end; ++tap) {
            // the first round passes: an empty stage's preceding phase is complete
            if (!tc::mbar_wait(&empty[s], parity)) {
                set_status(status, DEV_TIMEOUT);
                break;
            }
            uint8_t *a = smem + s * S::STAGE;
            tc::mbar_arrive_expect_tx(&full[s], S::A_BYTES + S::B_BYTES);
            load_tile(a, &xmap, &full[s], g, pos, dx, dy, dz);
            tc::bulk_load(a + S::A_BYTES, wpack + (size_t)tap * COUT * CIN, S::B_BYTES, &full[s]);
            if (++s == stages) {
                s = 0;
                parity ^= 1;
            }
            if (++dx == 2) {
                dx = -1;
                if (++dy == 2) {
                    dy = -1;
                    ++dz;
                }
            }
        }
    } else if (threadIdx.x == 32) {
        // MMA issuer
        constexpr uint32_t idesc = tc::idesc_bf16_f32(128, COUT);
        for (int it = 0, s = 0, parity = 0; it < tap_end - tap_begin; ++it) {
            if (!tc::mbar_wait(&full[s], parity)) {
                set_status(status, DEV_TIMEOUT);
                break;
            }
            tc::fence_after_sync();
            const uint32_t a = tc::smem_u32(smem + s * S::STAGE);
            const uint32_t b = a + S::A_BYTES;
#pragma unroll
            for (int kc = 0; kc < CIN / 16; ++kc) {
                const uint64_t ad = tc::smem_desc(a + kc * 2 * 2048, 2048, 128);
                const uint64_t bd = tc::smem_desc(b + kc * 2 * COUT * 16, COUT * 16, 128);
                tc::umma_bf16(tmem, ad, bd, idesc, (it > 0 || kc > 0) ? 1u : 0u);
            }
            tc::umma_commit(&empty[s]);
            if (++s == stages) {
                s = 0;
                parity ^= 1;
            }
        }
        tc::umma_commit(done);
    }

    // epilogue: thread = voxel (TMEM lane), 8 channels per TMEM load
    __syncwarp();  // lanes 0 of warps 0 and 1 rejoin after their producer / MMA roles
    const bool ready = tc::mbar_wait(done, 0);
    if (!ready && lane == 0) set_status(status, DEV_TIMEOUT);
    tc::fence_after_sync();
    const int m = warp * 32 + lane;
    const int plane = g.box_x * g.box_y;
    const int zz = m / plane, zn = pos.z0 + zz, r = m % plane;
    const int yy = pos.y0 + r / g.box_x, xx = pos.x0 + r % g.box_x;
    const bool stored = zz < pos.planes;  // false only past the last plane of a multi-plane tile
#pragma unroll
    for (int cb = 0; cb < COUT / 8; ++cb) {
        float v[8];
        tc::tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16) + cb * 8, v);
        if (!ready || !stored) continue;
        if (epi == EPI_BIAS_RELU) {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = fmaxf(v[q] + bias[cb * 8 + q], 0.0f);
        } else if (epi == EPI_MASK) {
            const uint4 mk = *reinterpret_cast<const uint4 *>(
                mask + ((((size_t)zn * g.mask_cg_total + g.mask_cg0 + cb) * g.H + yy) * g.W + xx) * 8);
            const __nv_bfloat16 *mb = reinterpret_cast<const __nv_bfloat16 *>(&mk);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __bfloat162float(mb[q]) > 0.0f ? v[q] : 0.0f;
        }
        if (y) {
            uint4 pk;
            __nv_bfloat162 *p2 = reinterpret_cast<__nv_bfloat162 *>(&pk);
#pragma unroll
            for (int q = 0; q < 4; ++q) p2[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
            *reinterpret_cast<uint4 *>(y + ((((size_t)zn * g.out_cg_total + g.out_cg0 + cb) * g.H + yy) * g.W + xx) * 8) =
                pk;
        }
        if (y_f32) {
            float *o = y_f32 + (((size_t)zn * g.H + yy) * g.W + xx) * COUT + cb * 8;
#pragma unroll
            for (int q = 0; q < 8; ++q) o[q] = v[q];
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

// ------------------------------------------------------------ weight grads
// Shared memory of wgrad_tc_kernel: a ring of stages, each holding the
// shifted x tiles of one group of TPG = 128 / CIN taps (the A operand, 128
// rows (tap, ci) of 2048-byte channel-group slabs, 32 KB) and the gz tile
// (B, COUT / 8 slabs).
template <int CIN, int COUT>
struct WgradSmem {
    static constexpr int TPG = 128 / CIN;                     // taps per MMA group
    static constexpr int NGROUPS = (27 + TPG - 1) / TPG;
    static constexpr int A_BYTES = 128 * 128 * 2;             // 16 slabs of 128 voxels x 16 B
    static constexpr int B_BYTES = COUT * 128 * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;           // a multiple of 2048
    static constexpr int STAGES = 4;
    static constexpr int BAR_OFF = STAGES * STAGE;
    static constexpr int BYTES = BAR_OFF + 128 + 1024;
    static constexpr int COLS_USED = NGROUPS * COUT;
    static constexpr int TMEM_COLS = COLS_USED <= 32 ? 32 : COLS_USED <= 64 ? 64 : COLS_USED <= 128 ? 128
                                   : COLS_USED <= 256 ? 256 : 512;
};

// dW[tap][co][ci] += sum over the voxels of tiles [t_begin, t_end) of
// gz[v][co] x[v + off(tap)][ci] (zero outside the sample), one CTA per
// chunk of tiles.  Per tile and tap group: warp 0 loads the group's
// shifted x tiles (the forward conv's TMA boxes; a plane outside its sample
// is zero fill) and the gz tile into a stage; thread 32 issues 8 MMAs (M = 128
// rows (tap, ci), N = COUT, K = 16 voxels, both operands MN-major) into
// the group's TMEM columns; at the end the four warps add their 128 lanes
// (rows) of every group to dw with atomics.
template <int CIN, int COUT>
__global__ void __launch_bounds__(CONV_THREADS)
wgrad_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap gmap, ConvGeom g,
                int tiles_per_cta, float *__restrict__ dw, int cin_store, int *status)
{
    using S = WgradSmem<CIN, COUT>;
    static_assert(CIN % 16 == 0 && 128 % CIN == 0 && COUT % 16 == 0 && S::COLS_USED <= 512, "wgrad shape");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + S::BAR_OFF);
    uint64_t *empty = full + S::STAGES;
    uint64_t *done = empty + S::STAGES;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntiles = g.tiles_x * g.tiles_y * g.tiles_z;
    const int t_begin = blockIdx.x * tiles_per_cta;
    const int t_end = min(ntiles, t_begin + tiles_per_cta);

    // rows of a partial last group read stale stage bytes: start them as zeros
    for (int q = threadIdx.x; q < S::STAGES * S::STAGE / 16; q += CONV_THREADS)
        reinterpret_cast<uint4 *>(smem)[q] = make_uint4(0, 0, 0, 0);
    if (warp == 0) {
        tc::tmem_alloc(tmem_slot, S::TMEM_COLS);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < S::STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(done, 1);
        tc::fence_mbar_init();
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the zeros before any TMA / MMA access
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // producers: a lane per tap of the group, and one for the gz tile
        int it = 0;
        bool ok = true;
        for (int t = t_begin; t < t_end && ok; ++t) {
            const TilePos pos = tile_pos(g, t);
            for (int gi = 0; gi < S::NGROUPS; ++gi, ++it) {
                const int s = it % S::STAGES;
                const int tap = gi * S::TPG + lane, ntap = min(S::TPG, 27 - gi * S::TPG);
                if (lane == 0) {
                    ok = it < S::STAGES || tc::mbar_wait(&empty[s], ((it / S::STAGES) - 1) & 1);
                    if (ok) tc::mbar_arrive_expect_tx(&full[s], ntap * CIN * 256 + COUT * 256);
                    else set_status(status, DEV_TIMEOUT);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                uint8_t *a = smem + s * S::STAGE;
                if (lane < ntap)
                    load_tile(a + lane * (CIN / 8) * 2048, &xmap, &full[s], g, pos, tap % 3 - 1,
                                       (tap / 3) % 3 - 1, tap / 9 - 1);
                else if (lane == 31)
                    load_tile(a + S::A_BYTES, &gmap, &full[s], g, pos, 0, 0, 0);
                __syncwarp();
            }
        }
    } else if (threadIdx.x == 32) {
        // MMA issuer
        constexpr uint32_t idesc = tc::idesc_bf16_f32(128, COUT, true);
        int it = 0;
        bool ok = true;
        for (int t = t_begin; t < t_end && ok; ++t) {
            for (int gi = 0; gi < S::NGROUPS; ++gi, ++it) {
                const int s = it % S::STAGES;
                if (!tc::mbar_wait(&full[s], (it / S::STAGES) & 1)) {
                    set_status(status, DEV_TIMEOUT);
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t a = tc::smem_u32(smem + s * S::STAGE);
                const uint32_t b = a + S::A_BYTES;
#pragma unroll
                for (int kc = 0; kc < 8; ++kc) {
                    // K = 16 voxels per MMA: the start moves by 16 voxels x 16 B
                    const uint64_t ad = tc::smem_desc(a + kc * 256, 128, 2048);
                    const uint64_t bd = tc::smem_desc(b + kc * 256, 128, 2048);
                    tc::umma_bf16(tmem + gi * COUT, ad, bd, idesc, (t > t_begin || kc > 0) ? 1u : 0u);
                }
                tc::umma_commit(&empty[s]);
            }
        }
        tc::umma_commit(done);
    }

    // epilogue: lane = row (tap, ci) of a group, 8 output channels per load
    __syncwarp();
    const bool ready = t_end > t_begin && tc::mbar_wait(done, 0);
    if (!ready && t_end > t_begin && lane == 0) set_status(status, DEV_TIMEOUT);
    tc::fence_after_sync();
    const int row = warp * 32 + lane;
    const int ci = row % CIN;
#pragma unroll 1
    for (int gi = 0; gi < S::NGROUPS; ++gi) {
        const int tap = gi * S::TPG + row / CIN;
#pragma unroll
        for (int cb = 0; cb < COUT / 8; ++cb) {
            float v[8];
            tc::tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16) + gi * COUT + cb * 8, v);
            if (!ready || tap >= 27 || ci >= cin_store) continue;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                atomicAdd(&dw[((size_t)tap * COUT + cb * 8 + q) * cin_store + ci], v[q]);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

// pack[tap][ci/8][co][ci%8] = w[tap][co][ci]   (forward), or with
// flip = 1 the weights of the backward-data convolution:
// pack[tap][co/8][ci][co%8] = w[26 - tap][co][ci].  The source holds
// cin_src <= cin input channels per (tap, co); the forward pack's channels
// ci >= cin_src are zero (a zero-padded input).  One launch makes all packs
// of the list (a network's 15 launches of 3 us were 5 % of a small training
// step); block b belongs to the job with first_block <= b.
__global__ void conv_pack_kernel(const __grid_constant__ PackList list)
{
    int j = 0;
    while (j + 1 < list.n && (int)blockIdx.x >= list.job[j + 1].first_block) ++j;
    const PackJob &job = list.job[j];
    const int cin = job.cin, cout = job.cout;
    const int n = 27 * cin * cout;
    const int q = (blockIdx.x - job.first_block) * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int tap = q / (cin * cout);
    const int r = q % (cin * cout);
    const int co = r / cin, ci = r % cin;
    const float v = ci < job.cin_src ? job.w[((size_t)tap * cout + co) * job.cin_src + ci] : 0.0f;
    size_t dst;
    if (!job.flip) {
        dst = (((size_t)tap * (cin / 8) + ci / 8) * cout + co) * 8 + ci % 8;
    } else {
        const int tp = 26 - tap;  // the packed conv has Cin' = cout, Cout' = cin
        dst = (((size_t)tp * (cout / 8) + co / 8) * cin + ci) * 8 + co % 8;
    }
    job.pack[dst] = __float2bfloat16_rn(v);
}

// dense FP32 (zn, y, x, C) <-> C8-blocked BF16
__global__ void to_blocked_kernel(const float *__restrict__ src, int NZ, int H, int W, int C,
                                  __nv_bfloat16 *__restrict__ dst, int cg_total, int cg0)
{
    const long long n = (long long)NZ * H * W * C;
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int c = (int)(q % C);
    long long v = q / C;
    const int x = (int)(v % W);
    v /= W;
    const int yy = (int)(v % H);
    const int zn = (int)(v / H);
    dst[((((size_t)zn * cg_total + cg0 + c / 8) * H + yy) * W + x) * 8 + c % 8] = __float2bfloat16_rn(src[q]);
}

__global__ void from_blocked_kernel(const __nv_bfloat16 *__restrict__ src, int NZ, int H, int W, int C, int cg_total,
                                    int cg0, float *__restrict__ dst)
{
    const long long n = (long long)NZ * H * W * C;
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int c = (int)(q % C);
    long long v = q / C;
    const int x = (int)(v % W);
    v /= W;
    const int yy = (int)(v % H);
    const int zn = (int)(v / H);
    dst[q] = __bfloat162float(src[((((size_t)zn * cg_total + cg0 + c / 8) * H + yy) * W + x) * 8 + c % 8]);
}

using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn()
{
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeFn)p;
    });
    return fn;
}

template <int CIN, int COUT>
gbsw_status launch_conv_t(const ConvCall &c, cudaStream_t s)
{
    using S = ConvSmem<CIN, COUT>;
    static bool configured = false;
    if (!configured) {
        GBSW_CUDA_TRY(cudaFuncSetAttribute(conv3d_tc_kernel<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           S::bytes(S::DEEP)));
        configured = true;
    }
    const int ntiles = c.geom.tiles_z * c.geom.tiles_y * c.geom.tiles_x;
    const int stages = ntiles <= sm_count() ? S::DEEP : S::STAGES;
    conv3d_tc_kernel<CIN, COUT><<<ntiles, CONV_THREADS, S::bytes(stages), s>>>(
        c.xmap, c.wpack, c.bias, c.y, c.y_f32, c.mask, c.geom, c.epi, stages, c.status);
    GBSW_LAUNCH_CHECK();
    return GBSW_OK;
}

template <int CIN, int COUT>
gbsw_status launch_wgrad_t(const WgradCall &c, cudaStream_t s)
{
    using S = WgradSmem<CIN, COUT>;
    static bool configured = false;
    if (!configured) {
        GBSW_CUDA_TRY(cudaFuncSetAttribute(wgrad_tc_kernel<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           S::BYTES));
        configured = true;
    }
    const int ntiles = c.geom.tiles_z * c.geom.tiles_y * c.geom.tiles_x;
    // one CTA per SM at most (the ring takes most of the shared memory); a
    // few tiles per CTA amortise the epilogue's atomics
    const int ctas = std::max(1, std::min(ntiles, sm_count()));
    const int per = ceil_div(ntiles, ctas);
    wgrad_tc_kernel<CIN, COUT><<<ceil_div(ntiles, per), CONV_THREADS, S::BYTES, s>>>(c.xmap, c.gmap, c.geom, per,
                                                                                     c.dw, c.cin_store, c.status);
    GBSW_LAUNCH_CHECK();
    return GBSW_OK;
}

}  // namespace

// Geometry of a conv over a C8-blocked tensor of NZ planes of H x W voxels.
gbsw_status conv_geometry(int NZ, int D, int H, int W, ConvGeom *g)
{
    if (NZ < 1 || D < 1 || NZ % D != 0 || H < 1 || W < 1) return GBSW_ERR_ARG;
    int bx = W >= 128 ? 128 : W;
    if (bx < 1 || 128 % bx != 0 || W % bx != 0) return GBSW_ERR_ARG;  // W a power of two or a multiple of 128
    int by = 128 / bx, bz = 1;
    if (H < by) {
        // small planes: the tile spans bz planes of H rows; boxes of >= 256 bytes
        if (by % H != 0 || bx * H < 16) return GBSW_ERR_ARG;
        bz = by / H;
        by = H;
    } else if (H % by != 0) {
        return GBSW_ERR_ARG;
    }
    // rows of at most 32 voxels, so that a box may be rows of voxels (LOAD_ROWS)
    if (bz == 1 && bx > 32 && H % 4 == 0) {
        bx = 32;
        by = 4;
    }
    g->load = bx > 32 ? LOAD_VOXELS : bz > 1 ? LOAD_SAMPLES : LOAD_ROWS;
    g->sample_tiles = bz > 1 && bz % D == 0 ? 0 : ceil_div(D, bz);
    g->NZ = NZ;
    g->D = D;
    g->H = H;
    g->W = W;
    g->box_x = bx;
    g->box_y = by;
    g->box_z = bz;
    g->tiles_x = W / bx;
    g->tiles_y = H / by;
    g->tiles_z = g->sample_tiles ? NZ / D * g->sample_tiles : ceil_div(NZ, bz);
    g->out_cg_total = g->out_cg0 = g->mask_cg_total = g->mask_cg0 = 0;
    return GBSW_OK;
}

// TMA map of a C8-blocked BF16 tensor with cg_total groups (all loaded).
gbsw_status conv_tensor_map(const __nv_bfloat16 *base, const ConvGeom &g, int cg_total, CUtensorMap *map)
{
    EncodeFn fn = encode_fn();
    if (!fn) return GBSW_ERR_CUDA;
    if (((uintptr_t)base & 15) != 0) return GBSW_ERR_ARG;
    const cuuint64_t W = g.W, H = g.H, D = g.D, NZ = g.NZ, cg = cg_total;
    const cuuint64_t row = W * 16, group = H * row, plane = cg * group;  // bytes
    const cuuint32_t bx = g.box_x, by = g.box_y, bz = g.box_z;
    const cuuint32_t bcg = cg_total;  // all channel groups at once
    cuuint64_t dims[5], strides[4];
    cuuint32_t box[5];
    auto set = [&](int k, cuuint64_t dim, cuuint64_t stride, cuuint32_t b) {
        dims[k] = dim;
        if (k > 0) strides[k - 1] = stride;
        box[k] = b;
    };
    switch (g.load) {
    case LOAD_VOXELS:
        set(0, 8, 0, 8);
        set(1, W, 16, bx);
        set(2, H, row, by);
        set(3, cg, group, bcg);
        set(4, NZ, plane, 1);
        break;
    case LOAD_ROWS:
        set(0, 8 * W, 0, 8 * bx);
        set(1, H, row, by);
        set(2, cg, group, bcg);
        set(3, NZ, plane, 1);
        set(4, 1, NZ * plane, 1);
        break;
    default: {
        const cuuint32_t planes = g.sample_tiles ? g.box_z : g.D;  // more than the sample has: zero fill
        set(0, 8 * W, 0, 8 * bx);
        set(1, H, row, by);
        set(2, D, plane, planes);
        set(3, NZ / D, D * plane, bz / planes);
        set(4, cg, group, bcg);
    }
    }
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void *)base, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? GBSW_OK : GBSW_ERR_ARG;
}

gbsw_status launch_conv(int cin, int cout, const ConvCall &c, cudaStream_t s)
{
#define CONV_CASE(A, B) \
    if (cin == A && cout == B) return launch_conv_t<A, B>(c, s);
    CONV_CASE(16, 16)
    CONV_CASE(16, 32)
    CONV_CASE(16, 64)
    CONV_CASE(32, 16)
    CONV_CASE(32, 32)
    CONV_CASE(32, 64)
    CONV_CASE(64, 16)
    CONV_CASE(64, 32)
#undef CONV_CASE
    return GBSW_ERR_ARG;
}

gbsw_status launch_wgrad_tc(int cin, int cout, const WgradCall &c, cudaStream_t s)
{
#define WG_CASE(A, B) \
    if (cin == A && cout == B) return launch_wgrad_t<A, B>(c, s);
    WG_CASE(16, 16)
    WG_CASE(16, 32)
    WG_CASE(32, 16)
    WG_CASE(32, 32)
    WG_CASE(32, 64)
    WG_CASE(64, 16)
    WG_CASE(64, 32)
#undef WG_CASE
    return GBSW_ERR_ARG;
}

gbsw_status pack_weights(PackList list, cudaStream_t s)
{
    if (list.n < 1 || list.n > PackList::MAX) return GBSW_ERR_ARG;
    int blocks = 0;
    for (int j = 0; j < list.n; ++j) {
        PackJob &job = list.job[j];
        if (job.cin_src < 1 || job.cin_src > job.cin || (job.flip && job.cin_src != job.cin)) return GBSW_ERR_ARG;
        job.first_block = blocks;
        blocks += ceil_div(27 * job.cin * job.cout, 256);
    }
    conv_pack_kernel<<<blocks, 256, 0, s>>>(list);
    GBSW_LAUNCH_CHECK();
    return GBSW_OK;
}

gbsw_status pack_weights(const float *w, int cin, int cout, int flip, __nv_bfloat16 *pack, cudaStream_t s)
{
    PackList list{};
    list.add(w, cin, cin, cout, flip, pack);
    return pack_weights(list, s);
}

gbsw_status to_blocked(const float *src, int NZ, int H, int W, int C, __nv_bfloat16 *dst, int cg_total, int cg0,
                       cudaStream_t s)
{
    const long long n = (long long)NZ * H * W * C;
    to_blocked_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, NZ, H, W, C, dst, cg_total, cg0);
    GBSW_LAUNCH_CHECK();
    return GBSW_OK;
}

gbsw_status from_blocked(const __nv_bfloat16 *src, int NZ, int H, int W, int C, int cg_total, int cg0, float *dst,
                         cudaStream_t s)
{
    const long long n = (long long)NZ * H * W * C;
    from_blocked_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, NZ, H, W, C, cg_total, cg0, dst);
    GBSW_LAUNCH_CHECK();
    return GBSW_OK;
}

}  // namespace gbsw
