// Learned warm start for value iteration: value iteration of a coarsened
// copy of each GridWorld (cells of 4 x 4 x 4 states) gives a coarse value
// per cell, and a fully convolutional 3-D network maps the cell features
// (mean reward of the non-obstacle states, obstacle fraction, largest
// terminal reward, -log(1 - gamma) / 5, the coarse value) to a correction of
// it; value iteration then starts from the corrected coarse values upsampled
// to the full grid. The solver is unchanged: a poor estimate only costs
// sweeps.
//
// Kernels (BF16 storage, FP32 accumulation, channels-last activations with
// 64 channels, "same" dilated 3 x 3 x 3 convolutions, tap t = (dz+1) * 9 +
// (dy+1) * 3 + (dx+1)):
//   conv_tma_kernel  y[v, n] = sum_t sum_k x[v + s d off(t), k] B_t[n, k] (+ b, ReLU, mask)
//                    on the tcgen05 tensor cores, operands by tensor copy:
//                    forward (s = +1, B_t[co, ci] = W[t, co, ci]) and data
//                    gradient (s = -1, B_t[ci, co] = W[t, co, ci], times the
//                    ReLU mask of the layer input)
//   conv_dw_tma_kernel  dW[t, co, ci] = sum_v dy[v, co] x[v + d off(t), ci], the voxels as the
//                    contraction of the same tensor cores (conv_dw_kernel: the SIMT
//                    form, for operands that no tensor copy can address)
//   plus features / targets / upsampling from a packed batch, the coarse
//   value iteration, the cell-level and full-grid loss gradients, Adam and
//   the FP32 -> BF16 weight casts.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "batch_internal.h"
#include "tc_common.cuh"

namespace cpmdp {

constexpr int kC = 64;        // channels of every activation
constexpr int kF = 4;         // coarsening factor per dimension

struct Dims {
    int n, z, y, x;           // instances and coarse grid
    __host__ __device__ int nvox() const { return n * z * y * x; }
};

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

constexpr int kCvBTile = 64 * 128;                   // one tap's weights: 64 channels x 64 bf16
constexpr long long kCvWaitCycles = 2000000000LL;    // about 1 s at 2 GHz

__device__ int g_conv_err = 0;

// Element offset of (row r, k) in a 64-wide bf16 tile with 128-byte rows
// and the 128-byte swizzle (16-byte chunk k / 8 of row r at chunk
// (k / 8) ^ (r % 8)).
__host__ __device__ __forceinline__ int sw_elem(int r, int k) { return r * 64 + ((((k >> 3) ^ (r & 7)) & 7) << 3) + (k & 7); }

// ---------------------------------------------------------------------------
// convolution (forward and data gradient): tiled tensor copies feed the
// tcgen05 tensor cores
//
// The same implicit GEMM. The output is cut into tiles of 128 voxels, a box
// of bx x by x bz voxels of one instance (tile row r = voxel
// (r / (bx by), (r / bx) % by, r % bx) of the box). A persistent CTA works
// through batches of 4 tiles whose accumulators (128 x 64 FP32 each) sit side
// by side in TMEM, twice over, so that the epilogue of one batch runs under
// the MMAs of the next. For each of the 9 tap groups (oz, ox) of a batch, the
// group's three weight tiles (oy = -1, 0, 1; pre-swizzled by the weight cast)
// arrive by bulk copy once for the 4 tiles, and each tile's input arrives by
// tensor copy of its box shifted by s d (oz, ., ox) (channels-last rows of
// 128 bytes, 128-byte swizzle: the K-major operand layout). In "tall" mode
// (one-plane tiles, bx a multiple of 8) one box of by + 2 d rows of y serves
// the group's three taps, which read it from row (s d oy + d) bx on (whole
// 1024-byte swizzle atoms); otherwise three boxes of the tile's own shape,
// one per oy, are copied. Voxels outside the grid arrive as zeros: the
// "same" padding. Roles: warp 4 issues the copies, one thread of warp 5 the
// MMAs (12 per tile and group: 3 taps x 4 K-steps of 16), warps 0-3 read the
// accumulators (thread = tile row = TMEM lane), apply bias and ReLU, or the
// ReLU mask of the layer input, and write bf16 rows (and FP32 channel 0).
// Every wait is bounded; one that runs out records an error (read by
// cpmdp_ws_sync) and stops every role, each after the copies and MMAs it
// issued have completed.

constexpr int kTmTiles = 4;                          // tiles (accumulators) per batch
constexpr uint32_t kTmCols = 2 * kTmTiles * 64;      // TMEM columns: two accumulator sets
constexpr int kTmThreads = 192;
constexpr int kTmBStage = 3 * kCvBTile;              // weight tiles of one tap group
constexpr int kTmBStages = 2;                        // weight ring
constexpr int kTmAMax = 3 * 128 * 128;               // largest input stage (three 128-row boxes)
constexpr int kTmMaxStages = 12;
constexpr int kTmSmemMax = 227 * 1024;

struct ConvGeo {
    int n, z, y, x;            // instances and grid
    int bx, by, bz;            // tile box
    int tx, ty, tz;            // tiles per dimension
    int tiles;
    int tall;                  // one (by + 2 dil)-row box per tap group
    int stage_bytes, stages;   // input ring
    int dil, sign, relu;
};

struct TmShared {
    uint64_t afull[kTmMaxStages], aempty[kTmMaxStages];
    uint64_t bfull[kTmBStages], bempty[kTmBStages], accf[2], acce[2];
    uint32_t tslot;
    int abort;
};

__device__ __forceinline__ bool tm_wait(uint64_t *bar, uint32_t phase, volatile int *abort) {
    const long long t0 = clock64();
    while (!tc::mbar_try(bar, phase)) {
        if (*abort) return false;
        if (clock64() - t0 > kCvWaitCycles) {
            *abort = 1;
            return false;
        }
    }
    return true;
}

// The same for a whole warp, which then goes on together.
__device__ __forceinline__ bool tm_wait_warp(uint64_t *bar, uint32_t phase, volatile int *abort) {
    return __all_sync(0xFFFFFFFFu, tm_wait(bar, phase, abort));
}

// A tile's place in the grid of tiles, stepped without dividing.
struct TileAt {
    int ix, iy, iz, n;
    template <typename Geo>
    __device__ __forceinline__ void set(const Geo &g, int tile) {
        ix = tile % g.tx; tile /= g.tx;
        iy = tile % g.ty; tile /= g.ty;
        iz = tile % g.tz;
        n = tile / g.tz;
    }
    template <typename Geo>
    __device__ __forceinline__ void add(const Geo &g, const TileAt &d) {
        ix += d.ix;
        int c = ix >= g.tx;
        ix -= c ? g.tx : 0;
        iy += d.iy + c;
        c = iy >= g.ty;
        iy -= c ? g.ty : 0;
        iz += d.iz + c;
        c = iz >= g.tz;
        iz -= c ? g.tz : 0;
        n += d.n + c;
    }
};

template <typename Geo>
__device__ __forceinline__ void tile_origin(const Geo &g, int tile, int &nn, int &x0, int &y0, int &z0) {
    int r = tile;
    const int ix = r % g.tx; r /= g.tx;
    const int iy = r % g.ty; r /= g.ty;
    const int iz = r % g.tz;
    nn = r / g.tz;
    x0 = ix * g.bx;
    y0 = iy * g.by;
    z0 = iz * g.bz;
}

__global__ void __launch_bounds__(kTmThreads, 1) conv_tma_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                const uint8_t *__restrict__ wimg,
                                                                const float *__restrict__ bias,
                                                                const __nv_bfloat16 *__restrict__ mask_act,
                                                                __nv_bfloat16 *__restrict__ y,
                                                                float *__restrict__ y0, ConvGeo g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sB = sm;
    uint8_t *sA = sm + kTmBStages * kTmBStage;
    TmShared &S = *reinterpret_cast<TmShared *>(sA + (size_t)g.stages * g.stage_bytes);
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        for (int i = 0; i < g.stages; i++) {
            tc::mbar_init(&S.afull[i], 1);
            tc::mbar_init(&S.aempty[i], 1);
        }
        for (int i = 0; i < kTmBStages; i++) {
            tc::mbar_init(&S.bfull[i], 1);
            tc::mbar_init(&S.bempty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            tc::mbar_init(&S.accf[i], 1);
            tc::mbar_init(&S.acce[i], 128);
        }
        S.abort = 0;
    }
    if (warp == 5) tc::tmem_alloc(&S.tslot, kTmCols);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tslot;
    volatile int *abort = &S.abort;
    const int nbatch = (g.tiles + kTmTiles - 1) / kTmTiles;
    const int d = g.dil, sg = g.sign;

    if (warp == 4) {
        // producer: weight tiles per tap group, input boxes per tile and group;
        // the warp runs the loop together, one thread issues
        const bool lead = tc::elect_lead();
        uint32_t as = 0, aph = 1, bs = 0, bph = 1;      // phase to wait for: the first round finds free slots
        uint32_t atotal = 0, btotal = 0;
        bool ok = true;
        const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
        const uint32_t abytes = g.tall ? (uint32_t)((g.by + 2 * d) * g.bx * 128) : 3u * 128u * 128u;
        TileAt at, one, hop;
        at.set(g, blockIdx.x * kTmTiles);
        one.set(g, 1);
        hop.set(g, gridDim.x * kTmTiles);
        for (int b = blockIdx.x; ok && b < nbatch; b += gridDim.x) {
            const int ntile = min(kTmTiles, g.tiles - b * kTmTiles);
            TileAt t4[kTmTiles];
            t4[0] = at;
#pragma unroll
            for (int j = 1; j < kTmTiles; j++) {
                t4[j] = t4[j - 1];
                t4[j].add(g, one);
            }
            at.add(g, hop);
            for (int grp = 0; ok && grp < 9; grp++) {
                const int oz = grp / 3 - 1, ox = grp % 3 - 1;
                if (btotal >= kTmBStages && !tm_wait_warp(&S.bempty[bs], bph, abort)) { ok = false; break; }
                tc::mbar_expect_tx_lead(lead, &S.bfull[bs], kTmBStage);
#pragma unroll
                for (int oy = 0; oy < 3; oy++)
                    tc::bulk_g2s_lead(lead, b0 + bs * kTmBStage + oy * kCvBTile,
                                      wimg + (size_t)((oz + 1) * 9 + oy * 3 + (ox + 1)) * kCvBTile, kCvBTile, &S.bfull[bs]);
                btotal++;
                if (++bs == kTmBStages) { bs = 0; bph ^= 1; }
#pragma unroll
                for (int j = 0; j < kTmTiles; j++) {
                    if (j >= ntile) break;
                    if (atotal >= (uint32_t)g.stages && !tm_wait_warp(&S.aempty[as], aph, abort)) { ok = false; break; }
                    const uint32_t dst = a0 + as * (uint32_t)g.stage_bytes;
                    const int xs = t4[j].ix * g.bx + sg * d * ox, ys = t4[j].iy * g.by, zs = t4[j].iz * g.bz + sg * d * oz;
                    tc::mbar_expect_tx_lead(lead, &S.afull[as], abytes);
                    if (g.tall) {
                        tc::tma_load_5d_lead(lead, dst, &tmx, 0, xs, ys - d, zs, t4[j].n, &S.afull[as]);
                    } else {
#pragma unroll
                        for (int oy = 0; oy < 3; oy++)
                            tc::tma_load_5d_lead(lead, dst + oy * 16384u, &tmx, 0, xs, ys + sg * d * (oy - 1), zs, t4[j].n,
                                                 &S.afull[as]);
                    }
                    atotal++;
                    if (++as == (uint32_t)g.stages) { as = 0; aph ^= 1; }
                }
            }
        }
        // every copy this warp issued lands before the CTA's shared memory
        // goes: the last of each slot was copy number total - 1 - back
        for (uint32_t back = 0; back < min(atotal, (uint32_t)g.stages); back++) {
            const uint32_t k = atotal - 1 - back;
            tc::mbar_wait(&S.afull[k % (uint32_t)g.stages], (k / (uint32_t)g.stages) & 1, kCvWaitCycles);
        }
        for (uint32_t back = 0; back < min(btotal, (uint32_t)kTmBStages); back++) {
            const uint32_t k = btotal - 1 - back;
            tc::mbar_wait(&S.bfull[k % kTmBStages], (k / kTmBStages) & 1, kCvWaitCycles);
        }
        __syncwarp();
    } else if (warp == 5) {
        // MMA issuer: the warp runs the loop together, one thread issues
        const bool lead = tc::elect_lead();
        uint32_t as = 0, aph = 0, bs = 0, bph = 0, bcount = 0;
        uint64_t *lastbar = nullptr;
        uint32_t lastph = 0;
        bool ok = true;
        const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
        const uint32_t ostep = g.tall ? (uint32_t)(sg * d * g.bx * 128) : 16384u;   // from one oy to the next
        const uint32_t ofirst = g.tall ? (uint32_t)((d - sg * d) * g.bx * 128) : 0u;
        for (int b = blockIdx.x; ok && b < nbatch; b += gridDim.x, bcount++) {
            const uint32_t buf = bcount & 1;
            if (bcount >= 2 && !tm_wait_warp(&S.acce[buf], ((bcount >> 1) - 1) & 1, abort)) { ok = false; break; }
            tc::fence_after();
            const uint32_t dacc = tmem + buf * (kTmCols / 2);
            const int ntile = min(kTmTiles, g.tiles - b * kTmTiles);
            for (int grp = 0; ok && grp < 9; grp++) {
                if (!tm_wait_warp(&S.bfull[bs], bph, abort)) { ok = false; break; }
                const uint64_t bd = tc::sdesc(b0 + bs * kTmBStage);
                for (int j = 0; j < ntile; j++) {
                    if (!tm_wait_warp(&S.afull[as], aph, abort)) { ok = false; break; }
                    tc::fence_after();
                    const uint64_t ad = tc::sdesc(a0 + as * (uint32_t)g.stage_bytes + ofirst);
                    const uint32_t dj = dacc + (uint32_t)j * 64u, acc0 = grp > 0 ? 1u : 0u;
#pragma unroll
                    for (int oy = 0; oy < 3; oy++)
#pragma unroll
                        for (int ks = 0; ks < 4; ks++)
                            tc::mma_lead(lead, dj, ad + (uint64_t)(((int)ostep * oy + ks * 32) >> 4),
                                         bd + (uint64_t)((oy * kCvBTile + ks * 32) >> 4), tc::kIdescM128N64,
                                         oy > 0 || ks > 0 ? 1u : acc0);
                    tc::commit_lead(lead, &S.aempty[as]);
                    lastbar = &S.aempty[as];
                    lastph = aph;
                    if (++as == (uint32_t)g.stages) { as = 0; aph ^= 1; }
                }
                if (!ok) break;
                tc::commit_lead(lead, &S.bempty[bs]);
                lastbar = &S.bempty[bs];
                lastph = bph;
                if (++bs == kTmBStages) { bs = 0; bph ^= 1; }
            }
            if (!ok) break;
            tc::commit_lead(lead, &S.accf[buf]);
            lastbar = &S.accf[buf];
            lastph = (bcount >> 1) & 1;
        }
        // the MMAs complete in order: the last commit covers them all
        if (lastbar) tc::mbar_wait(lastbar, lastph, kCvWaitCycles);
        __syncwarp();
    } else {
        // epilogue: warps 0-3, thread = tile row = TMEM lane
        const int r = tid;
        const int xl = r % g.bx, yl = (r / g.bx) % g.by, zl = r / (g.bx * g.by);
        uint32_t bcount = 0;
        for (int b = blockIdx.x; b < nbatch; b += gridDim.x, bcount++) {
            const int buf = bcount & 1;
            const bool okw = tm_wait(&S.accf[buf], (bcount >> 1) & 1, abort);
            if (!__all_sync(0xFFFFFFFFu, okw)) break;
            tc::fence_after();
            for (int j = 0; j < kTmTiles; j++) {
                const int tile = b * kTmTiles + j;
                if (tile >= g.tiles) break;
                int nn, x0, y0t, z0;
                tile_origin(g, tile, nn, x0, y0t, z0);
                float acc[64];
                tc::tmem_ld64(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)buf * (kTmCols / 2) + (uint32_t)j * 64u,
                              acc);
                const int gx = x0 + xl, gy = y0t + yl, gz = z0 + zl;
                if (gx < g.x && gy < g.y && gz < g.z) {
                    const size_t v = ((size_t)(nn * g.z + gz) * g.y + gy) * g.x + gx;
#pragma unroll
                    for (int c = 0; c < 64; c++) acc[c] += bias ? bias[c] : 0.f;
                    if (mask_act) {
                        const uint4 *mrow = reinterpret_cast<const uint4 *>(mask_act + v * kC);
#pragma unroll
                        for (int q = 0; q < 8; q++) {
                            const uint4 m = mrow[q];
                            const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                            for (int h = 0; h < 8; h++) {
                                const uint16_t bits = (uint16_t)(w[h >> 1] >> (16 * (h & 1)));
                                if (!(bf(__ushort_as_bfloat16(bits)) > 0.f)) acc[8 * q + h] = 0.f;
                            }
                        }
                    }
                    uint4 *dst = reinterpret_cast<uint4 *>(y + v * kC);
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        uint32_t w[4];
#pragma unroll
                        for (int h = 0; h < 4; h++) {
                            float a0 = acc[8 * q + 2 * h], a1 = acc[8 * q + 2 * h + 1];
                            if (g.relu) { a0 = fmaxf(a0, 0.f); a1 = fmaxf(a1, 0.f); }
                            if (q == 0 && h == 0 && y0) y0[v] = a0;
                            w[h] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a0)) |
                                   ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a1)) << 16);
                        }
                        dst[q] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
            tc::fence_before();
            tc::mbar_arrive(&S.acce[buf]);
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0 && S.abort) atomicExch(&g_conv_err, 1);
    if (warp == 5) tc::tmem_dealloc(tmem, kTmCols);
}

// ---------------------------------------------------------------------------
// weight gradient on the tensor cores
//
// dW[t] is a 64 x 64 product contracted over all voxels, for 27 taps that read
// the same dy and shifted copies of the same x. A CTA takes one (oz, ox) and
// every splits-th tile of 128 voxels; the tile's dy and its shifted x arrive
// by tensor copy (tall mode: one box of by + 2 d rows of y serves the three oy
// taps; otherwise three boxes). Channels-last voxel rows are MN-major operands
// as they lie, so nothing is transposed: A stacks two taps' 64 input channels
// (two 64-wide MN atoms, the leading byte offset being the distance between
// the taps' rows: oy = -1 and 0, then 0 again and 1), B is dy, K = 128 voxels.
// The tensor cores truncate when they add to an accumulator, so a long chain
// of them drifts (1.7e-6 off at 131,072 voxels when each CTA kept its sums in
// TMEM to the end, 3.0e-7 on the FP32 pipe): each tile's sums (8 steps) are
// drained and added up in registers, round to nearest, while the next tile
// runs in another TMEM accumulator. At the end the CTA adds its sums to dW
// with coalesced reductions.
// A voxel of a tile beyond the grid has dy = 0 from the copy: it adds 0 x,
// which is 0 unless x is infinite or a NaN there. So in a grid that is no
// multiple of the tile (RAGGED), a thread whose sums come out not finite takes
// them again over the voxels in the grid (dw_again). It looks once, at the end
// (30.8 us at 30 x 9^3 as without it, 39 us with a look at every tile's sums),
// in an instance of its own (its registers cost 32 x 16^3 a microsecond).
// One layer at 32 x 16^3 voxels: 1,660 us on the FP32 pipe (conv_dw_kernel),
// 47 us here; the x and dy copies run at 7 TB/s from L2. One CTA for all nine
// taps of an oz with its sums kept in TMEM took 38 us, at the error above.
//
// Error against FP64, root mean square over the largest outputs' scale, of
// positive x (after a ReLU): the truncation inside a tile leaves about 7e-8
// whatever the size, every reduction into dW a rounding of the whole sum. The
// FP32 pipe, 512 voxels a block, is at its best with few blocks (6.3e-8 at
// 4,096 voxels, 8.9e-8 at 16,384, 24e-8 at 131,072; this kernel as above
// 9.3e-8, 9.4e-8, 9.7e-8). So below kDwFew voxels a tile's 8 steps go to two
// accumulators (half the truncation), up to kDwFewer voxels with at most 8
// reductions an output, and less than one tile of voxels stays on the FP32
// pipe: 5.9e-8 at 2,048 voxels (FP32 pipe 6.6e-8), 6.0e-8 at 4,096, 6.1e-8 at
// 8,192 (6.9e-8), 7.2e-8 at 16,384. It costs time: 8.4 us for 6.6 at 4,096
// voxels, 12.5 for 10.6 at 16,384, and would 55 for 47 at 131,072, where the
// longer chain of register additions gains nothing either.
constexpr uint32_t kDwIdesc = tc::kIdescM128N64AMN | (1u << 16);   // A and B MN-major
constexpr int kDwMaxStages = 6;
constexpr int kDwFew = 24576, kDwFewer = 8192;       // voxels (see above)
constexpr int kDwAccMax = 4;                         // accumulators (128 TMEM columns each) in turn: two tiles'

struct DwGeo {
    int n, z, y, x;
    int bx, by, bz, tx, ty, tz, tiles, splits;
    int tall, dil;
    int xbytes, bstep;         // bytes of a tile's x boxes, between the rows of two oy
    int stage_bytes, stages;
};

struct DwShared {
    uint64_t full[kDwMaxStages], empty[kDwMaxStages], accf[kDwAccMax], acce[kDwAccMax];
    uint32_t tslot;
    int abort;
};

// What a drain thread adds to dW for one tap (its input channel ci, all output
// channels), on the FP32 pipe and without the voxels beyond the grid.
__device__ __noinline__ void dw_again(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ dy,
                                      float *__restrict__ dw, const DwGeo &g, int split, int oz, int oy, int ox, int ci) {
    float *o = dw + (size_t)((oz + 1) * 9 + (oy + 1) * 3 + ox + 1) * kC * kC + ci;
    for (int co0 = 0; co0 < kC; co0 += 32) {
        float sum[32];
#pragma unroll
        for (int c = 0; c < 32; c++) sum[c] = 0.f;
        for (int tile = split; tile < g.tiles; tile += g.splits) {
            int nn, x0, y0, z0;
            tile_origin(g, tile, nn, x0, y0, z0);
            float v[32];
#pragma unroll
            for (int c = 0; c < 32; c++) v[c] = 0.f;
            for (int r = 0; r < 128; r++) {
                const int xx = x0 + r % g.bx, yy = y0 + r / g.bx % g.by, zz = z0 + r / g.bx / g.by;
                if (xx >= g.x || yy >= g.y || zz >= g.z) continue;
                const long long x2 = xx + (long long)g.dil * ox, y2 = yy + (long long)g.dil * oy,
                                z2 = zz + (long long)g.dil * oz, plane = (long long)nn * g.z;
                const bool in = x2 >= 0 && x2 < g.x && y2 >= 0 && y2 < g.y && z2 >= 0 && z2 < g.z;
                const float xv = in ? bf(x[(((plane + z2) * g.y + y2) * g.x + x2) * kC + ci]) : 0.f;
                const uint4 *d = reinterpret_cast<const uint4 *>(dy + (((plane + zz) * g.y + yy) * g.x + xx) * kC + co0);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint4 m = d[q];
                    const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        v[8 * q + 2 * k] = fmaf(__uint_as_float(w[k] << 16), xv, v[8 * q + 2 * k]);
                        v[8 * q + 2 * k + 1] = fmaf(__uint_as_float(w[k] & 0xFFFF0000u), xv, v[8 * q + 2 * k + 1]);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 32; c++) sum[c] += v[c];
        }
#pragma unroll
        for (int c = 0; c < 32; c++) atomicAdd(o + (co0 + c) * kC, sum[c]);
    }
}

// PARTS: accumulators a tile's 8 steps are spread over. (A wait that runs out
// leaves its role's loops by goto: a flag in their conditions cost 4 %.)
template <int PARTS, bool RAGGED>
__global__ void __launch_bounds__(kTmThreads, 1) conv_dw_tma_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                    const __grid_constant__ CUtensorMap tmd,
                                                                    const __nv_bfloat16 *__restrict__ x,
                                                                    const __nv_bfloat16 *__restrict__ dy,
                                                                    float *__restrict__ dw,
                                                                    const __grid_constant__ DwGeo g) {
    constexpr int kDwAcc = 2 * PARTS;
    static_assert(kDwAcc <= kDwAccMax, "TMEM columns");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    DwShared &S = *reinterpret_cast<DwShared *>(sm + (size_t)g.stages * g.stage_bytes);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int split = blockIdx.x / 9, oz = (int)(blockIdx.x % 9) / 3 - 1, ox = (int)(blockIdx.x % 3) - 1;
    if (tid == 0) {
        for (int i = 0; i < g.stages; i++) {
            tc::mbar_init(&S.full[i], 1);
            tc::mbar_init(&S.empty[i], 1);
        }
        for (int i = 0; i < kDwAcc; i++) {
            tc::mbar_init(&S.accf[i], 1);
            tc::mbar_init(&S.acce[i], 128);
        }
        S.abort = 0;
    }
    if (warp == 5) tc::tmem_alloc(&S.tslot, 128 * kDwAcc);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tslot;
    volatile int *abort = &S.abort;
    const int d = g.dil;

    if (warp == 4) {
        const bool lead = tc::elect_lead();
        uint32_t st = 0, ph = 1, total = 0;              // the first round finds free slots
        const uint32_t s0 = tc::smem_u32(sm);
        TileAt at, hop;
        at.set(g, split);
        hop.set(g, g.splits);
        for (int tile = split; tile < g.tiles; tile += g.splits) {
            if (total >= (uint32_t)g.stages && !tm_wait_warp(&S.empty[st], ph, abort)) break;
            const uint32_t dst = s0 + st * (uint32_t)g.stage_bytes;
            const int x0 = at.ix * g.bx, y0 = at.iy * g.by, z0 = at.iz * g.bz, xs = x0 + d * ox, zs = z0 + d * oz;
            tc::mbar_expect_tx_lead(lead, &S.full[st], (uint32_t)g.xbytes + 16384u);
            if (g.tall) {
                tc::tma_load_5d_lead(lead, dst, &tmx, 0, xs, y0 - d, zs, at.n, &S.full[st]);
            } else {
#pragma unroll
                for (int oy = 0; oy < 3; oy++)
                    tc::tma_load_5d_lead(lead, dst + (uint32_t)(oy * g.bstep), &tmx, 0, xs, y0 + d * (oy - 1), zs, at.n,
                                         &S.full[st]);
            }
            tc::tma_load_5d_lead(lead, dst + (uint32_t)g.xbytes, &tmd, 0, x0, y0, z0, at.n, &S.full[st]);
            at.add(g, hop);
            total++;
            if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1; }
        }
        // every copy this warp issued lands before the CTA's shared memory goes
        for (uint32_t back = 0; back < min(total, (uint32_t)g.stages); back++) {
            const uint32_t k = total - 1 - back;
            tc::mbar_wait(&S.full[k % (uint32_t)g.stages], (k / (uint32_t)g.stages) & 1, kCvWaitCycles);
        }
        __syncwarp();
    } else if (warp == 5) {
        const bool lead = tc::elect_lead();
        uint32_t count = 0, st = 0, sph = 0;
        uint64_t *lastbar = nullptr;
        uint32_t lastph = 0;
        const uint32_t s0 = tc::smem_u32(sm);
        for (int tile = split; tile < g.tiles; tile += g.splits) {
            const uint32_t a0 = s0 + st * (uint32_t)g.stage_bytes;
            const uint64_t ad = tc::sdesc_mn(a0, (uint32_t)g.bstep), bd = tc::sdesc_mn(a0 + (uint32_t)g.xbytes, 8192u);
#pragma unroll
            for (int part = 0; part < PARTS; part++, count++) {
                const uint32_t buf = count % kDwAcc;
                if (count >= kDwAcc && !tm_wait_warp(&S.acce[buf], (count / kDwAcc - 1) & 1, abort)) goto issued;
                if (part == 0 && !tm_wait_warp(&S.full[st], sph, abort)) goto issued;
                tc::fence_after();
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int n = 0; n < 8 / PARTS; n++) {
                        const int ks = part * (8 / PARTS) + n;
                        tc::mma_lead(lead, tmem + 128u * buf + 64u * i, ad + (uint64_t)((i * g.bstep + ks * 2048) >> 4),
                                     bd + (uint64_t)(ks * 2048 >> 4), kDwIdesc, n > 0 ? 1u : 0u);
                    }
                if (part == PARTS - 1) tc::commit_lead(lead, &S.empty[st]);
                tc::commit_lead(lead, &S.accf[buf]);
                lastbar = &S.accf[buf];
                lastph = (count / kDwAcc) & 1;
            }
            if (++st == (uint32_t)g.stages) { st = 0; sph ^= 1; }
        }
    issued:
        // the MMAs complete in order: the last commit covers them all
        if (lastbar) tc::mbar_wait(lastbar, lastph, kCvWaitCycles);
        __syncwarp();
    } else {
        const int half = tid >> 6, ci = tid & 63;   // rows of A: 64 of oy = -1 (i = 1: 0), 64 of oy = 0 (1)
        const uint32_t t0 = tmem + ((uint32_t)(32 * warp) << 16);
        float acc[2][kC];
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int c = 0; c < kC; c++) acc[i][c] = 0.f;
        bool ok = true;
        uint32_t count = 0;
        for (int tile = split; tile < g.tiles; tile += g.splits) {
#pragma unroll
            for (int part = 0; part < PARTS; part++, count++) {
                const int buf = count % kDwAcc;
                ok = __all_sync(0xFFFFFFFFu, tm_wait(&S.accf[buf], (count / kDwAcc) & 1, abort));
                if (!ok) goto drained;
                tc::fence_after();
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    if (i == 1 && half == 0) continue;   // oy = 0 again (whole warps)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        float v[32];
                        tc::tmem_ld32(t0 + 128u * buf + 64u * i + 32u * h, v);
#pragma unroll
                        for (int c = 0; c < 32; c++) acc[i][32 * h + c] += v[c];
                    }
                }
                tc::fence_before();
                tc::mbar_arrive(&S.acce[buf]);
            }
        }
    drained:
        if (RAGGED && ok) {
            float z[4] = {0.f, 0.f, 0.f, 0.f};       // stays 0, or a NaN where a sum is not finite
#pragma unroll
            for (int c = 0; c < 2 * kC; c++) z[c & 3] = fmaf(acc[c / kC][c % kC], 0.f, z[c & 3]);
            if (isnan((z[0] + z[1]) + (z[2] + z[3]))) {
                for (int i = 0; i < 1 + half; i++) dw_again(x, dy, dw, g, split, oz, i + half - 1, ox, ci);
                ok = false;                          // added
            }
        }
        if (ok) {
#pragma unroll
            for (int i = 0; i < 2; i++) {
                if (i == 1 && half == 0) continue;
                float *o = dw + (size_t)((oz + 1) * 9 + (i + half) * 3 + ox + 1) * kC * kC + ci;
#pragma unroll
                for (int co = 0; co < kC; co++) atomicAdd(o + co * kC, acc[i][co]);
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0 && S.abort) atomicExch(&g_conv_err, 1);
    if (warp == 5) tc::tmem_dealloc(tmem, 128 * kDwAcc);
}

// The same on the FP32 pipe, for operands that are not 16-byte aligned and for
// less than a tile of voxels:
// dW[t, co, ci] += sum over a chunk of voxels of dy[v, co] x[v + d off(t), ci]
__global__ void __launch_bounds__(256) conv_dw_kernel(const __nv_bfloat16 *__restrict__ x,
                                                      const __nv_bfloat16 *__restrict__ dy, float *__restrict__ dw,
                                                      Dims dm, int dil, int chunk) {
    __shared__ float sD[32][65];   // [voxel][co]
    __shared__ float sX[32][65];   // [voxel][ci]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int t = blockIdx.y;
    const int oz = dil * (t / 9 - 1), oy = dil * ((t / 3) % 3 - 1), ox = dil * (t % 3 - 1);
    const int nvox = dm.nvox();
    const int vbeg = blockIdx.x * chunk, vend = min(vbeg + chunk, nvox);
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0.f;
    for (int vb = vbeg; vb < vend; vb += 32) {
        for (int e = tid; e < 32 * 64; e += 256) {
            const int vv = e >> 6, c = e & 63;
            const int v = vb + vv;
            float dv = 0.f, xv = 0.f;
            if (v < vend) {
                dv = bf(dy[(size_t)v * kC + c]);
                int r = v;
                const int xx = r % dm.x; r /= dm.x;
                const int yy = r % dm.y; r /= dm.y;
                const int zz = r % dm.z; const int nn = r / dm.z;
                const int z2 = zz + oz, y2 = yy + oy, x2 = xx + ox;
                if (z2 >= 0 && z2 < dm.z && y2 >= 0 && y2 < dm.y && x2 >= 0 && x2 < dm.x)
                    xv = bf(x[((size_t)((nn * dm.z + z2) * dm.y + y2) * dm.x + x2) * kC + c]);
            }
            sD[vv][c] = dv;
            sX[vv][c] = xv;
        }
        __syncthreads();
#pragma unroll 8
        for (int vv = 0; vv < 32; vv++) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; i++) a[i] = sD[vv][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; j++) b[j] = sX[vv][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            atomicAdd(&dw[(size_t)t * kC * kC + (ty + 16 * i) * kC + tx + 16 * j], acc[i][j]);
}

// db[c] += sum_v dy[v, c], 16 bytes (8 channels) a load: 8 lanes a voxel, 32
// voxels a block at a time. Bound by the read of dy; one 2-byte load a thread
// (conv_db_kernel) took 37 us for 131,072 voxels.
__global__ void __launch_bounds__(256) conv_db_vec_kernel(const uint4 *__restrict__ dy, float *__restrict__ db, int nvox) {
    __shared__ float sh[8][kC];
    const int q = threadIdx.x & 7, warp = threadIdx.x >> 5;
    float s[8];
#pragma unroll
    for (int k = 0; k < 8; k++) s[k] = 0.f;
#pragma unroll 4
    for (int v = blockIdx.x * 32 + (threadIdx.x >> 3); v < nvox; v += gridDim.x * 32) {
        const uint4 m = dy[(size_t)v * 8 + q];
        const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            s[2 * k] += __uint_as_float(w[k] << 16);
            s[2 * k + 1] += __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
        s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], 8);
        s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], 16);
    }
    if ((threadIdx.x & 31) < 8) {
#pragma unroll
        for (int k = 0; k < 8; k++) sh[warp][8 * q + k] = s[k];
    }
    __syncthreads();
    if (threadIdx.x < kC) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; w++) t += sh[w][threadIdx.x];
        atomicAdd(&db[threadIdx.x], t);
    }
}

// The same for a dy that is not 16-byte aligned.
__global__ void conv_db_kernel(const __nv_bfloat16 *__restrict__ dy, float *__restrict__ db, int nvox) {
    const int c = threadIdx.x & 63, lane_group = threadIdx.x >> 6;   // 4 groups of 64 threads
    float s = 0.f;
    for (int v = blockIdx.x * 4 + lane_group; v < nvox; v += gridDim.x * 4) s += bf(dy[(size_t)v * kC + c]);
    atomicAdd(&db[c], s);
}

// dy[v, 0] = 2 (pred - target) mask / nvox, other channels 0; loss += sum mask (pred - target)^2 / nvox
__global__ void loss_grad_kernel(const float *__restrict__ pred, const float *__restrict__ target,
                                 const float *__restrict__ mask, __nv_bfloat16 *__restrict__ dy, float *loss, int nvox) {
    __shared__ float sh[8];
    float l = 0.f;
    const float inv = 1.f / (float)nvox;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nvox; v += gridDim.x * blockDim.x) {
        const float d = (pred[v] - target[v]) * mask[v];
        l += d * d * inv;
        dy[(size_t)v * kC] = __float2bfloat16_rn(2.f * d * inv);
#pragma unroll 4
        for (int c = 1; c < kC; c++) dy[(size_t)v * kC + c] = __float2bfloat16_rn(0.f);
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[w];
        if (loss) atomicAdd(loss, s);
    }
}

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// W [t][co][ci] (FP32) -> per tap the B tiles of the tensor-core convolution
// (64 rows x 64 bf16, 128-byte swizzle): wf row co, column ci (forward) and
// wb row ci, column co (data gradient).
__global__ void cast_weights_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wf,
                                    __nv_bfloat16 *__restrict__ wb, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long t = i / (kC * kC), r = i % (kC * kC);
        const int co = (int)(r / kC), ci = (int)(r % kC);
        const __nv_bfloat16 h = __float2bfloat16_rn(w[i]);
        wf[t * kC * kC + sw_elem(co, ci)] = h;
        wb[t * kC * kC + sw_elem(ci, co)] = h;
    }
}

// ---------------------------------------------------------------------------
// batch <-> coarse grids (instances first .. first + count - 1, equal shapes)

__device__ __forceinline__ void coarse_of(const BatchInst &I, int cell, int &cz, int &cy, int &cx, int &zc, int &yc,
                                          int &xc) {
    zc = (I.shape[0] + kF - 1) / kF;
    yc = (I.shape[1] + kF - 1) / kF;
    xc = (I.shape[2] + kF - 1) / kF;
    cx = cell % xc;
    cy = (cell / xc) % yc;
    cz = cell / (xc * yc);
}

// The 4 states of a cell's row are taken without branching per state (the
// terminals, a handful in an instance, apart): code bits 6 and 7 of the four
// bytes at once, and a zero added for a state that does not count.
struct RowSums {
    int n = 0, obst = 0, free = 0, any_t = 0;
    float rfree = 0.f, rlive = 0.f, tmax = 0.f;   // rewards of free states, of all but obstacles
    __device__ __forceinline__ void add(const float (&r)[kF], unsigned cw, int states) {
        const unsigned o = cw & 0x40404040u, t = cw & 0x80808080u;
        n += states;
        obst += __popc(o);
        free += states - __popc(o | t);
#pragma unroll
        for (int k = 0; k < kF; k++) {
            const float live = (o >> (8 * k) & 0xFFu) ? 0.f : r[k];
            rlive += live;
            rfree += (t >> (8 * k) & 0xFFu) ? 0.f : live;
        }
        if (t) {
#pragma unroll
            for (int k = 0; k < kF; k++)
                if (t >> (8 * k) & 0xFFu) {
                    tmax = any_t ? fmaxf(tmax, r[k]) : r[k];
                    any_t = 1;
                }
        }
    }
};

// The rows of coarse cell (cz, cy, cx) of instance I: one 16-byte reward load
// and one 4-byte code load where the row is a full aligned group of 4, which
// it is in every instance whose x side is a multiple of 4. A state outside the
// grid counts for nothing (code 0, reward 0, not among `states`).
__device__ __forceinline__ RowSums cell_sums(const BatchInst &I, const uint8_t *__restrict__ code,
                                             const float *__restrict__ R, int cz, int cy, int cx) {
    RowSums s;
    const int x0 = cx * kF, nx = min(kF, I.shape[2] - x0);
    const bool vec = I.shape[2] % 4 == 0 && I.offset % 4 == 0;
    for (int z = cz * kF; z < min((cz + 1) * kF, I.shape[0]); z++) {
#pragma unroll
        for (int j = 0; j < kF; j++) {
            const int y = cy * kF + j;
            if (y >= I.shape[1]) break;
            const long long at = I.offset + (long long)z * I.stride[0] + (long long)y * I.stride[1] + x0;
            float r[kF];
            unsigned cw = 0;
            if (vec) {
                const float4 rv = *reinterpret_cast<const float4 *>(R + at);
                cw = *reinterpret_cast<const unsigned *>(code + at);
                r[0] = rv.x; r[1] = rv.y; r[2] = rv.z; r[3] = rv.w;
            } else {
#pragma unroll
                for (int k = 0; k < kF; k++) {
                    r[k] = k < nx ? R[at + k] : 0.f;
                    cw |= (unsigned)(k < nx ? code[at + k] : 0) << (8 * k);
                }
            }
            s.add(r, cw, nx);
        }
    }
    return s;
}

constexpr int kFeatThreads = 256;

// One thread per coarse cell (blockIdx.y: instances); rows of the cell whose x
// extent is a full aligned group of 4 (every row of an instance with x side a
// multiple of 4) are read as one 16-byte reward load and one 4-byte code load,
// so neighbouring cells' threads read neighbouring bytes. A cell's 128 bytes
// of channels are written by 8 threads, 16 bytes each, from shared memory: a
// warp stores whole lines. Bound by the memory (168 MB read, 67 MB written for
// 128 instances of 64^3: 35 us) and the loads in flight: 78 us with one thread
// writing a cell's channels, 51 us so.
__global__ void __launch_bounds__(kFeatThreads) features_kernel(const BatchInst *__restrict__ inst,
                                                                const uint8_t *__restrict__ code,
                                                                const float *__restrict__ R, int first, int count,
                                                                int cells, __nv_bfloat16 *__restrict__ feat) {
    __shared__ uint2 sh[kFeatThreads];
    const int base = blockIdx.x * kFeatThreads, cell = base + threadIdx.x;
    for (int i = blockIdx.y; i < count; i += gridDim.y) {
        if (cell < cells) {
            const BatchInst I = inst[first + i];
            int cz, cy, cx, zc, yc, xc;
            coarse_of(I, cell, cz, cy, cx, zc, yc, xc);
            const RowSums c = cell_sums(I, code, R, cz, cy, cx);
            const int live = c.n - c.obst;
            const __nv_bfloat162 lo = __halves2bfloat162(__float2bfloat16_rn(live ? c.rlive / live : 0.f),
                                                         __float2bfloat16_rn((float)c.obst / (float)c.n));
            const __nv_bfloat162 hi = __halves2bfloat162(__float2bfloat16_rn(c.any_t ? c.tmax : 0.f),
                                                         __float2bfloat16_rn(-logf(1.f - I.gamma) / 5.f));
            sh[threadIdx.x] = make_uint2(*reinterpret_cast<const unsigned *>(&lo), *reinterpret_cast<const unsigned *>(&hi));
        }
        __syncthreads();
        // channels 4..63: zero (channel 4 is the coarse value, written later)
        uint4 *out = reinterpret_cast<uint4 *>(feat + ((size_t)i * cells + base) * kC);
        const int part = min(kFeatThreads, cells - base) * 8;
        for (int e = threadIdx.x; e < part; e += kFeatThreads) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if ((e & 7) == 0) { v.x = sh[e >> 3].x; v.y = sh[e >> 3].y; }
            out[e] = v;
        }
        __syncthreads();
    }
}

__global__ void targets_kernel(const BatchInst *__restrict__ inst, const uint8_t *__restrict__ code,
                               const float *__restrict__ V, int first, int count, int cells,
                               const float *__restrict__ base, float *__restrict__ target, float *__restrict__ mask) {
    const long long total = (long long)count * cells;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total; g += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(g / cells), cell = (int)(g % cells);
        const BatchInst I = inst[first + i];
        int cz, cy, cx, zc, yc, xc;
        coarse_of(I, cell, cz, cy, cx, zc, yc, xc);
        const unsigned ob = 1u << (2 * I.ndim);
        float s = 0.f;
        int live = 0;
        for (int z = cz * kF; z < min((cz + 1) * kF, I.shape[0]); z++)
            for (int y = cy * kF; y < min((cy + 1) * kF, I.shape[1]); y++)
                for (int x = cx * kF; x < min((cx + 1) * kF, I.shape[2]); x++) {
                    const long long st = I.offset + (long long)z * I.stride[0] + y * I.stride[1] + x;
                    if (code[st] & ob) continue;
                    live++;
                    s += V[st];
                }
        target[g] = (live ? s / live : 0.f) - (base ? base[g] : 0.f);
        mask[g] = live ? 1.f : 0.f;
    }
}

// Interpolation in one dimension: the coarse values sit at the cell centres, a
// fine coordinate p at (p + 0.5) / 4 - 0.5 in cell units, clamped to the
// outermost centres.
// Weight of cell c of nc at its fine coordinate 4 c - 2 + o, 0 <= o < 8: the
// clamp gives an outermost cell all of the coordinates beyond its centre.
__device__ __forceinline__ float cell_weight(int o, int c, int nc) {
    const float w = 0.125f + 0.25f * (float)(o < 4 ? o : 7 - o);
    return (c == 0 && o < 4) || (c == nc - 1 && o >= 4) ? 1.f : w;
}

__device__ __forceinline__ float lerp(float a, float b, float t) { return (1.f - t) * a + t * b; }

// Trilinear interpolation of coarse + base at half the states of a coarse cell,
// its rows y = 4 cy + 2 half and the next: 4 x 2 x 4 states. They lie between
// the centres cz - 1, cz, cz + 1 and cx - 1, cx, cx + 1, and between two centres
// in y, so 18 cell values, reduced over y, then z, then x, serve all 32 (state
// by state: 256 loads and products; a whole cell a thread: too many registers
// for enough warps).
struct Patch {
    float c[3][2][3];          // z, y, x: coarse + base
    float tz[4], ty[2], tx[4]; // weights of the upper centre (1: the lower one is the same)
    __device__ __forceinline__ static void weights(int c, int nc, float (&t)[4]) {
        t[0] = c > 0 ? 0.625f : 1.f;
        t[1] = c > 0 ? 0.875f : 1.f;
        t[2] = c < nc - 1 ? 0.125f : 0.f;
        t[3] = c < nc - 1 ? 0.375f : 0.f;
    }
    __device__ __forceinline__ void load(int cz, int cy, int half, int cx, int zc, int yc, int xc, const float *cv,
                                         const float *bv) {
        float t[4];
        weights(cz, zc, tz);
        weights(cy, yc, t);
        weights(cx, xc, tx);
        ty[0] = half ? t[2] : t[0];
        ty[1] = half ? t[3] : t[1];
        const int x[3] = {max(cx - 1, 0), cx, min(cx + 1, xc - 1)}, z[3] = {max(cz - 1, 0), cz, min(cz + 1, zc - 1)};
        const int y[2] = {half ? cy : max(cy - 1, 0), half ? min(cy + 1, yc - 1) : cy};
#pragma unroll
        for (int m = 0; m < 3; m++)
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int r = (z[m] * yc + y[i]) * xc;
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    c[m][i][j] = cv[r + x[j]];
                    if (bv) c[m][i][j] += bv[r + x[j]];
                }
            }
    }
    // row g of the two in all planes, reduced over y (g, h known at compile time)
    __device__ __forceinline__ void plane(int g, float (&e)[3][3]) const {
#pragma unroll
        for (int m = 0; m < 3; m++)
#pragma unroll
            for (int j = 0; j < 3; j++) e[m][j] = lerp(c[m][0][j], c[m][1][j], ty[g]);
    }
    // its four states of plane z = 4 cz + h
    __device__ __forceinline__ void row(const float (&e)[3][3], int h, float (&v)[4]) const {
        float f[3];
#pragma unroll
        for (int j = 0; j < 3; j++) f[j] = lerp(e[h < 2 ? 0 : 1][j], e[h < 2 ? 1 : 2][j], tz[h]);
#pragma unroll
        for (int k = 0; k < 4; k++) v[k] = lerp(f[k < 2 ? 0 : 1], f[k < 2 ? 1 : 2], tx[k]);
    }
};

// Coarse estimate (plus base) upsampled to every fine state: free states
// take the interpolation, terminals R(t), obstacles 0. One thread per half
// cell (blockIdx.y: instances); rows whose length is a multiple of 4 (16-byte
// aligned, as every instance starts on a multiple of 4 states) are written in
// 16-byte stores. Bound by the stores (V 4 B, code 1 B a state, 25 us) and the
// instructions; 128 instances of 64^3: 208 us state by state, 54 us so.
__global__ void __launch_bounds__(128) upsample_kernel(const BatchInst *__restrict__ inst, const uint8_t *__restrict__ code,
                                                       const float *__restrict__ R, int first, int count, int cells,
                                                       const float *__restrict__ coarse, const float *__restrict__ base,
                                                       float *__restrict__ V) {
    const BatchInst &I0 = inst[first];
    const int Z = I0.shape[0], Y = I0.shape[1], X = I0.shape[2];
    const int zc = (Z + kF - 1) / kF, yc = (Y + kF - 1) / kF, xc = (X + kF - 1) / kF;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= 2 * cells) return;
    const int row = id / xc, cx = id - row * xc, cz = row / (2 * yc), hy = row - cz * 2 * yc, cy = hy >> 1, half = hy & 1;
    const unsigned ob = 1u << 6, tb = 1u << 7;   // 3-D codes
    const bool full = X % 4 == 0;
    const int live = min(4, X - 4 * cx);
    for (int i = blockIdx.y; i < count; i += gridDim.y) {
        Patch pt;
        pt.load(cz, cy, half, cx, zc, yc, xc, coarse + (long long)i * cells, base ? base + (long long)i * cells : nullptr);
        const long long at = inst[first + i].offset + (long long)(4 * cz * Y + 2 * hy) * X + 4 * cx;
#pragma unroll
        for (int g = 0; g < 2; g++) {
            if (2 * hy + g >= Y) break;
            float e[3][3];
            pt.plane(g, e);
            unsigned cw[4];
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const long long s0 = at + ((long long)h * Y + g) * X;
                cw[h] = 0;
                if (4 * cz + h >= Z) continue;
                if (full) cw[h] = *reinterpret_cast<const unsigned *>(code + s0);
                else
                    for (int k = 0; k < 4; k++) cw[h] |= (unsigned)(k < live ? code[s0 + k] : ob) << (8 * k);
            }
#pragma unroll
            for (int h = 0; h < 4; h++) {
                if (4 * cz + h >= Z) break;
                const long long s0 = at + ((long long)h * Y + g) * X;
                float v[4];
                pt.row(e, h, v);
                if (cw[h] & 0xC0C0C0C0u) {
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const unsigned c = cw[h] >> (8 * k);
                        if (c & ob) v[k] = 0.f;
                        else if (c & tb) v[k] = R[s0 + k];
                    }
                }
                if (full) {
                    *reinterpret_cast<float4 *>(V + s0) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        if (k < live) V[s0 + k] = v[k];
                }
            }
        }
    }
}

// Fine-level loss of a coarse estimate: with Vh = upsample(base + pred),
// r(s) = Vh(s) - Vt(s) on the free states (0 on terminals and obstacles,
// where the upsampling is exact); loss += sum r^2 * inv. Threads as in
// upsample_kernel. 32 instances of 64^3 (75 MB, 11 us): 123 us with one state a
// thread, 30 us so.
__global__ void __launch_bounds__(128) fine_resid_kernel(const BatchInst *__restrict__ inst, const uint8_t *__restrict__ code,
                                                         int first, int count, int cells, const float *__restrict__ pred,
                                                         const float *__restrict__ base, const float *__restrict__ Vt,
                                                         float *__restrict__ r, float inv, float *loss) {
    __shared__ float sh[8];
    const BatchInst &I0 = inst[first];
    const int Z = I0.shape[0], Y = I0.shape[1], X = I0.shape[2];
    const int zc = (Z + kF - 1) / kF, yc = (Y + kF - 1) / kF, xc = (X + kF - 1) / kF;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = id / xc, cx = id - row * xc, cz = row / (2 * yc), hy = row - cz * 2 * yc, cy = hy >> 1, half = hy & 1;
    const bool on = id < 2 * cells;
    const bool full = X % 4 == 0, vt16 = full && (reinterpret_cast<uintptr_t>(Vt) & 15) == 0,
               r16 = full && (reinterpret_cast<uintptr_t>(r) & 15) == 0;   // a multiple of 4 states an instance
    const int live = min(4, X - 4 * cx);
    float l = 0.f;
    for (int i = blockIdx.y; on && i < count; i += gridDim.y) {
        Patch pt;
        pt.load(cz, cy, half, cx, zc, yc, xc, pred + (long long)i * cells, base ? base + (long long)i * cells : nullptr);
        const long long at = (long long)(4 * cz * Y + 2 * hy) * X + 4 * cx, off = inst[first + i].offset;
        float *ri = r + (long long)i * I0.nstates;
#pragma unroll
        for (int g = 0; g < 2; g++) {
            if (2 * hy + g >= Y) break;
            float e[3][3];
            pt.plane(g, e);
#pragma unroll
            for (int h = 0; h < 4; h++) {
                if (4 * cz + h >= Z) break;
                const long long s0 = at + ((long long)h * Y + g) * X;
                unsigned cw = 0;
                float vt[4] = {0.f, 0.f, 0.f, 0.f}, d[4];
                if (full) cw = *reinterpret_cast<const unsigned *>(code + off + s0);
                else
                    for (int k = 0; k < 4; k++) cw |= (unsigned)(k < live ? code[off + s0 + k] : 0x40u) << (8 * k);
                if (vt16) {
                    const float4 v = *reinterpret_cast<const float4 *>(Vt + off + s0);
                    vt[0] = v.x; vt[1] = v.y; vt[2] = v.z; vt[3] = v.w;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        if (k < live) vt[k] = Vt[off + s0 + k];
                }
                pt.row(e, h, d);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    d[k] = (cw >> (8 * k) & 0xC0u) ? 0.f : d[k] - vt[k];
                    l += d[k] * d[k] * inv;
                }
                if (r16) {
                    *reinterpret_cast<float4 *>(ri + s0) = make_float4(d[0], d[1], d[2], d[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        if (k < live) ri[s0 + k] = d[k];
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) sum += sh[w];
        if (loss) atomicAdd(loss, sum);
    }
}

// Gradient of that loss with respect to the coarse estimate: the transpose
// of the interpolation, dL/dpred(c) = 2 inv sum_s w(s, c) r(s) over the fine
// states whose interpolation reads cell c (coordinates 4c - 2 .. 4c + 5 in
// each dimension); written into channel 0 of dy, the other channels 0.
// One thread a cell, its sum in the order z, y, x (the result is rounded to
// bf16, where another order shows as a whole last place). A block takes 16 x 16
// cells of one cz; the fine plane under them comes to shared memory by
// asynchronous copies, one plane ahead of the sums, each state once, and a cell
// reads a row's 8 states as three 16-byte pieces. Bound by those reads (192 a
// cell). 32 instances of 64^3: 173 us with every thread reading its states from
// global memory, 39 us so (17 us with the sums taken dimension by dimension,
// which moved 6e-7 of the gradients by a last place of bf16).
// A cell's channels are written in 16-byte stores where dy lies so, else one by one.
constexpr int kGradCells = 16;                       // cells of a tile per dimension
constexpr int kGradRows = kF * kGradCells + 4;       // fine rows under it: 4 cy0 - 2 ..
constexpr int kGradPitch = kF * kGradCells + 8;      // fine states of a row: 4 cx0 - 4 ..
__global__ void __launch_bounds__(kGradCells *kGradCells) fine_grad_kernel(const BatchInst *__restrict__ inst, int first,
                                                                          int count, int zc, int yc, int xc,
                                                                          const float *__restrict__ r, float inv,
                                                                          __nv_bfloat16 *__restrict__ dy) {
    __shared__ __align__(16) float plane[2][kGradRows * kGradPitch];
    const BatchInst &I0 = inst[first];
    const int Z = I0.shape[0], Y = I0.shape[1], X = I0.shape[2];
    const int xt = (xc + kGradCells - 1) / kGradCells, yt = (yc + kGradCells - 1) / kGradCells;
    const int cz = blockIdx.x / (xt * yt), rest = blockIdx.x - cz * xt * yt;
    const int cy0 = rest / xt * kGradCells, cx0 = (rest - rest / xt * xt) * kGradCells;
    const int lx = threadIdx.x % kGradCells, ly = threadIdx.x / kGradCells, cx = cx0 + lx, cy = cy0 + ly;
    const int x0 = kF * cx0 - 4, y0 = kF * cy0 - 2, zlo = max(0, kF * cz - 2), zhi = min(Z - 1, kF * cz + 5);
    for (int i = blockIdx.y; i < count; i += gridDim.y) {
        const float *ri = r + (long long)i * I0.nstates;
        auto fetch = [&](int z) {
            float *p = plane[z & 1];
            const float *src = ri + (long long)z * Y * X;
            for (int e = threadIdx.x; e < kGradRows * kGradPitch; e += kGradCells * kGradCells) {
                const int row = e / kGradPitch, y = y0 + row, x = x0 + e - row * kGradPitch;
                if (y >= 0 && y < Y && x >= 0 && x < X)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(p + e)),
                                 "l"(src + (long long)y * X + x)
                                 : "memory");
                else
                    p[e] = 0.f;
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(zlo);
        float acc = 0.f;
        for (int z = zlo; z <= zhi; z++) {
            if (z < zhi) {
                fetch(z + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();                         // plane z is there, for every thread
            const float wz = cell_weight(z - (kF * cz - 2), cz, zc);
            const float *p = plane[z & 1] + kF * ly * kGradPitch + kF * lx;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const float wzy = wz * cell_weight(j, cy, yc);
                float v[12];
#pragma unroll
                for (int q = 0; q < 3; q++) {
                    const float4 f = *reinterpret_cast<const float4 *>(p + j * kGradPitch + 4 * q);
                    v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
                }
#pragma unroll
                for (int k = 0; k < 8; k++) acc = fmaf(wzy * cell_weight(k, cx, xc), v[k + 2], acc);
            }
            __syncthreads();                         // and read: its buffer takes plane z + 2
        }
        if (cx < xc && cy < yc) {
            __nv_bfloat16 *d = dy + ((((size_t)i * zc + cz) * yc + cy) * xc + cx) * kC;
            const __nv_bfloat16 grad = __float2bfloat16_rn(2.f * inv * acc);
            if ((reinterpret_cast<uintptr_t>(dy) & 15) == 0) {
                uint4 w = make_uint4((unsigned)__bfloat16_as_ushort(grad), 0u, 0u, 0u);
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    reinterpret_cast<uint4 *>(d)[q] = w;
                    w.x = 0u;
                }
            } else {
                d[0] = grad;
#pragma unroll 4
                for (int c = 1; c < kC; c++) d[c] = __float2bfloat16_rn(0.f);
            }
        }
    }
}

// Value iteration of a coarsened copy of each instance, one CTA per
// instance, entirely in shared memory (the input feature that gives the
// network a view of the whole grid). Coarse cell = 4 x 4 x 4 fine states:
// an obstacle when at least half of its states are obstacles, else a
// terminal of value max R(t) when it holds terminals, else a free cell whose
// reward per coarse step is the mean fine reward of its free states times
// 1 + gamma + gamma^2 + gamma^3 (four fine steps); discount gamma^4, the
// instance's slip model, walls and obstacle cells block moves. Jacobi sweeps
// from zero until max |dV| < tol or max_sweeps.
constexpr int kCoarseThreads = 1024;
constexpr int kMaxCoarseCells = 8192;

template <int N>
__global__ void __launch_bounds__(kCoarseThreads) coarse_vi_kernel(const BatchInst *__restrict__ inst,
                                                                   const uint8_t *__restrict__ code,
                                                                   const float *__restrict__ R, int first, int cells,
                                                                   float tol, int max_sweeps,
                                                                   float *__restrict__ coarse_v,
                                                                   __nv_bfloat16 *__restrict__ feat) {
    extern __shared__ uint8_t smem_raw[];
    float *va = reinterpret_cast<float *>(smem_raw);                 // V (even sweeps)
    float *vb = va + cells;                                          // V (odd sweeps)
    float *rsum = vb + cells;                                        // coarse reward
    uint8_t *kind = reinterpret_cast<uint8_t *>(rsum + cells);      // bits 0-5 blocked moves, 6 obstacle, 7 terminal
    const int tid = threadIdx.x;
    const int i = blockIdx.x;
    const BatchInst I = inst[first + i];
    const int zc = (I.shape[0] + kF - 1) / kF, yc = (I.shape[1] + kF - 1) / kF, xc = (I.shape[2] + kF - 1) / kF;
    const float g = I.gamma;
    // gamma^4 and 1 + gamma + gamma^2 + gamma^3 (the rounding spelled out, as below)
    const float g3 = __fmul_rn(__fmul_rn(g, g), g);
    const float gc = __fmul_rn(g3, g), steps = __fadd_rn(__fmaf_rn(g, g, __fadd_rn(1.f, g)), g3);
    for (int c = tid; c < cells; c += kCoarseThreads) {
        const int cz = c / (yc * xc), cy = (c / xc) % yc, cx = c % xc;
        const RowSums sums = cell_sums(I, code, R, cz, cy, cx);
        uint8_t k = 0;
        float r = 0.f;
        if (2 * sums.obst >= sums.n) k = 0x40;
        else if (sums.any_t) { k = 0x80; r = sums.tmax; }
        else r = sums.free ? sums.rfree / (float)sums.free * steps : 0.f;
        kind[c] = k;
        rsum[c] = r;
    }
    __syncthreads();
    for (int c = tid; c < cells; c += kCoarseThreads) {
        const int cz = c / (yc * xc), cy = (c / xc) % yc, cx = c % xc;
        uint8_t k = kind[c];
        const int nbr[6] = {cz > 0 ? c - yc * xc : -1, cz < zc - 1 ? c + yc * xc : -1, cy > 0 ? c - xc : -1,
                            cy < yc - 1 ? c + xc : -1, cx > 0 ? c - 1 : -1, cx < xc - 1 ? c + 1 : -1};
#pragma unroll
        for (int j = 0; j < 6; j++)
            if (nbr[j] < 0 || (kind[nbr[j]] & 0x40)) k |= (uint8_t)(1u << j);
        kind[c] = k;
        const float v0 = (k & 0x80) ? rsum[c] : 0.f;
        va[c] = v0;
        vb[c] = v0;
    }
    __syncthreads();
    // Each thread keeps the kinds and rewards of its cells in registers (N
    // cells, kCoarseThreads apart, so a cell's neighbours are at fixed offsets
    // from the thread's); the larger of a dimension's two neighbours gives the
    // larger of its two actions' values (weights >= 0, rounding is monotone).
    // 128 instances of 64^3: 165 us with every cell's kind, reward and
    // addresses worked out on each sweep, 512 threads and a branch per fine
    // state; 93 us so.
    const float wm = I.w_move, wp = I.w_perp;
    const int s0 = yc * xc, s1 = xc;
    float rr[N];
    unsigned kk[(N + 3) / 4];
#pragma unroll
    for (int n = 0; n < (N + 3) / 4; n++) kk[n] = 0;
#pragma unroll
    for (int n = 0; n < N; n++) {
        const int c = tid + n * kCoarseThreads;
        rr[n] = c < cells ? rsum[c] : 0.f;
        kk[n / 4] |= (c < cells ? (unsigned)kind[c] : 0x40u) << (8 * (n % 4));
    }
    float *src = va, *dst = vb;
    for (int sweep = 0; sweep < max_sweeps; sweep++) {
        int open = 0;
        const float *p = src + tid, *zm = p - s0, *zp = p + s0, *ym = p - s1, *yp = p + s1;
        float *out = dst + tid;
#pragma unroll
        for (int n = 0; n < N; n++) {
            const unsigned k = kk[n / 4] >> (8 * (n % 4));
            if (k & 0xC0u) continue;   // obstacles (0) and terminals (their value) never change
            const int o = n * kCoarseThreads;
            const float self = p[o];
            const float n0 = (k & 1u) ? self : zm[o], n1 = (k & 2u) ? self : zp[o], n2 = (k & 4u) ? self : ym[o];
            const float n3 = (k & 8u) ? self : yp[o], n4 = (k & 16u) ? self : p[o - 1], n5 = (k & 32u) ? self : p[o + 1];
            const float P0 = n0 + n1, P1 = n2 + n3, P2 = n4 + n5;
            // (the rounding spelled out: the values go on as bf16 features)
            float best = __fmaf_rn(wm, fmaxf(n0, n1), __fmul_rn(wp, P1 + P2));
            best = fmaxf(best, __fmaf_rn(wm, fmaxf(n2, n3), __fmul_rn(wp, P0 + P2)));
            best = fmaxf(best, __fmaf_rn(wm, fmaxf(n4, n5), __fmul_rn(wp, P0 + P1)));
            const float v = rr[n] + gc * best;
            out[o] = v;
            open |= fabsf(v - self) >= tol;
        }
        float *t = src; src = dst; dst = t;
        if (!__syncthreads_or(open)) break;
    }
    for (int c = tid; c < cells; c += kCoarseThreads) {
        const uint8_t k = kind[c];
        const float v = (k & 0x40) ? 0.f : src[c];
        coarse_v[(long long)i * cells + c] = v;
        if (feat) feat[((long long)i * cells + c) * kC + 4] = __float2bfloat16_rn(v);
    }
}

static int grid_for(long long n, int per_block) {
    long long g = (n + per_block - 1) / per_block;
    if (g > 65535LL * 16) g = 65535LL * 16;
    return (int)(g < 1 ? 1 : g);
}

// Shape check shared by the batch <-> coarse calls: instances first..first+count-1
// must be 3-D and of one shape (each is addressed through its own offset in
// the packed layout); returns the coarse cell count.
static cpmdp_status batch_range(const cpmdp_batch *B, int first, int count, int *cells) {
    if (!B || count < 1 || first < 0 || first + count > B->ninst) { set_error("instance range outside the batch"); return CPMDP_EINVAL; }
    const BatchInst &I0 = B->inst[(size_t)first];
    if (I0.ndim != 3) { set_error("the warm start takes 3-D instances"); return CPMDP_EINVAL; }
    for (int i = first; i < first + count; i++) {
        const BatchInst &I = B->inst[(size_t)i];
        if (I.ndim != 3 || I.shape[0] != I0.shape[0] || I.shape[1] != I0.shape[1] || I.shape[2] != I0.shape[2]) {
            set_error("instances %d..%d must share one shape", first, first + count - 1);
            return CPMDP_EINVAL;
        }
    }
    *cells = ((I0.shape[0] + kF - 1) / kF) * ((I0.shape[1] + kF - 1) / kF) * ((I0.shape[2] + kF - 1) / kF);
    return CPMDP_OK;
}

// cuTensorMapEncodeTiled from the driver, looked up once.
static PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            (void)cudaGetLastError();
    }
    return fn;
}

static int pow2_at_least(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Tiles of 128 voxels: a box of bx x by x bz.
template <typename Geo>
static bool tile_shape(const Dims &dm, int dil, Geo &g) {
    g.n = dm.n; g.z = dm.z; g.y = dm.y; g.x = dm.x;
    g.bx = std::min(16, std::max(8, pow2_at_least(dm.x)));
    g.by = std::min(128 / g.bx, pow2_at_least(dm.y));
    g.bz = 128 / (g.bx * g.by);
    g.tx = (dm.x + g.bx - 1) / g.bx;
    g.ty = (dm.y + g.by - 1) / g.by;
    g.tz = (dm.z + g.bz - 1) / g.bz;
    const long long tiles = (long long)g.tx * g.ty * g.tz * dm.n;
    if (tiles > (1LL << 30)) return false;
    g.tiles = (int)tiles;
    g.tall = g.bz == 1 && g.bx % 8 == 0 && g.by + 2LL * dil <= 256 && (g.by + 2LL * dil) * g.bx * 128 <= kTmAMax;
    g.dil = dil;
    return true;
}

// Tensor map of a channels-last activation, boxes of 64 channels x bx x rows x bz.
static cudaError_t act_map(const __nv_bfloat16 *x, const Dims &dm, int bx, int rows, int bz, CUtensorMap *map) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t gdim[5] = {(cuuint64_t)kC, (cuuint64_t)dm.x, (cuuint64_t)dm.y, (cuuint64_t)dm.z, (cuuint64_t)dm.n};
    const cuuint64_t gstride[4] = {(cuuint64_t)kC * 2, (cuuint64_t)kC * 2 * dm.x, (cuuint64_t)kC * 2 * dm.x * dm.y,
                                   (cuuint64_t)kC * 2 * dm.x * dm.y * dm.z};
    const cuuint32_t box[5] = {(cuuint32_t)kC, (cuuint32_t)bx, (cuuint32_t)rows, (cuuint32_t)bz, 1u};
    const cuuint32_t estride[5] = {1u, 1u, 1u, 1u, 1u};
    if (enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16 *>(x), gdim, gstride, box, estride,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

// Tile shape, input ring and tensor map of one convolution launch.
static cudaError_t launch_conv(const __nv_bfloat16 *x, const uint8_t *wimg, const float *bias,
                               const __nv_bfloat16 *mask_act, __nv_bfloat16 *y, float *y0, Dims dm, int dil, int sign,
                               int relu, cudaStream_t st) {
    ConvGeo g;
    if (!tile_shape(dm, dil, g)) return cudaErrorInvalidValue;
    const int tall_rows = (g.by + 2 * dil) * g.bx;
    g.stage_bytes = g.tall ? ((tall_rows * 128 + 1023) & ~1023) : kTmAMax;
    g.stages = std::min(kTmMaxStages,
                        (kTmSmemMax - 1024 - kTmBStages * kTmBStage - (int)sizeof(TmShared)) / g.stage_bytes);
    g.sign = sign;
    g.relu = relu;
    const size_t smem = 1024 + (size_t)kTmBStages * kTmBStage + (size_t)g.stages * g.stage_bytes + sizeof(TmShared);

    CUtensorMap map;
    cudaError_t e = act_map(x, dm, g.bx, g.tall ? g.by + 2 * dil : g.by, g.bz, &map);
    if (e != cudaSuccess) return e;

    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(conv_tma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTmSmemMax)) !=
        cudaSuccess)
        return e;
    const int nbatch = (g.tiles + kTmTiles - 1) / kTmTiles;
    const int grid = std::max(1, std::min(nbatch, sms));
    conv_tma_kernel<<<grid, kTmThreads, smem, st>>>(map, wimg, bias, mask_act, y, y0, g);
    return cudaGetLastError();
}

// Weight gradient on the tensor cores; cudaErrorNotSupported where no tensor
// copy can address the operands, or there is less than one tile of voxels.
static cudaError_t launch_dw(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *dw, Dims dm, int dil, cudaStream_t st) {
    if (((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dy)) & 15) || dm.nvox() < 128) return cudaErrorNotSupported;
    DwGeo g;
    if (!tile_shape(dm, dil, g)) return cudaErrorNotSupported;
    const int rows = g.by + 2 * dil;
    g.bstep = g.tall ? dil * g.bx * 128 : 16384;
    g.xbytes = g.tall ? rows * g.bx * 128 : 3 * 16384;   // whole 1024-byte atoms: bx is a multiple of 8
    g.stage_bytes = g.xbytes + 16384;
    g.stages = std::min(kDwMaxStages, (kTmSmemMax - 1024 - (int)sizeof(DwShared)) / g.stage_bytes);
    if (g.stages < 1) return cudaErrorNotSupported;
    CUtensorMap mx, md;
    cudaError_t e = act_map(x, dm, g.bx, g.tall ? rows : g.by, g.bz, &mx);
    if (e == cudaSuccess) e = act_map(dy, dm, g.bx, g.by, g.bz, &md);
    if (e != cudaSuccess) return cudaErrorNotSupported;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const bool ragged = dm.x % g.bx || dm.y % g.by || dm.z % g.bz;
    const auto kern = dm.nvox() < kDwFew ? (ragged ? conv_dw_tma_kernel<2, true> : conv_dw_tma_kernel<2, false>)
                                         : (ragged ? conv_dw_tma_kernel<1, true> : conv_dw_tma_kernel<1, false>);
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTmSmemMax)) != cudaSuccess) return e;
    g.splits = std::max(1, std::min(g.tiles, sms / 9));
    if (dm.nvox() <= kDwFewer) g.splits = std::min(g.splits, 8);
    const size_t smem = 1024 + (size_t)g.stages * g.stage_bytes + sizeof(DwShared);
    kern<<<9 * g.splits, kTmThreads, smem, st>>>(mx, md, x, dy, dw, g);
    return cudaGetLastError();
}

static cpmdp_status dims_ok(int n, int z, int y, int x, int dil) {
    if (n < 1 || z < 1 || y < 1 || x < 1 || dil < 1 || (long long)n * z * y * x > (1LL << 31) - 64) {
        set_error("invalid convolution dimensions");
        return CPMDP_EINVAL;
    }
    return CPMDP_OK;
}

}  // namespace cpmdp

using namespace cpmdp;

extern "C" {

cpmdp_status cpmdp_ws_features(const cpmdp_batch *B, int32_t first, int32_t count, uint16_t *feat, void *stream) {
    int cells = 0;
    cpmdp_status s = batch_range(B, first, count, &cells);
    if (s != CPMDP_OK) return s;
    const dim3 grid((cells + kFeatThreads - 1) / kFeatThreads, std::min(count, 65535));
    features_kernel<<<grid, kFeatThreads, 0, (cudaStream_t)stream>>>(B->d_inst, B->d_code, B->d_R, first, count, cells,
                                                                     (__nv_bfloat16 *)feat);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_targets(const cpmdp_batch *B, const float *V, int32_t first, int32_t count, const float *base,
                              float *target, float *mask, void *stream) {
    int cells = 0;
    cpmdp_status s = batch_range(B, first, count, &cells);
    if (s != CPMDP_OK) return s;
    const long long n = (long long)count * cells;
    targets_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(B->d_inst, B->d_code, V, first, count, cells,
                                                                       base, target, mask);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_upsample(const cpmdp_batch *B, const float *coarse, const float *base, int32_t first,
                               int32_t count, float *V, void *stream) {
    int cells = 0;
    cpmdp_status s = batch_range(B, first, count, &cells);
    if (s != CPMDP_OK) return s;
    const BatchInst &I0 = B->inst[(size_t)first];
    const dim3 grid((unsigned)((2LL * cells + 127) / 128), (unsigned)std::min(count, 65535));
    upsample_kernel<<<grid, 128, 0, (cudaStream_t)stream>>>(B->d_inst, B->d_code, B->d_R, first, count, cells, coarse,
                                                            base, V);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_fine_loss_grad(const cpmdp_batch *B, const float *V_target, int32_t first, int32_t count,
                                     const float *pred, const float *base, float *resid, uint16_t *dy, float *loss,
                                     void *stream) {
    int cells = 0;
    cpmdp_status s = batch_range(B, first, count, &cells);
    if (s != CPMDP_OK) return s;
    if (!V_target || !pred || !resid || !dy) { set_error("V_target, pred, resid and dy are required"); return CPMDP_EINVAL; }
    const long long n = (long long)count * B->inst[(size_t)first].nstates;
    const float inv = (float)(1.0 / (double)n);
    const BatchInst &I0 = B->inst[(size_t)first];
    const int zc = (I0.shape[0] + kF - 1) / kF, yc = (I0.shape[1] + kF - 1) / kF, xc = (I0.shape[2] + kF - 1) / kF;
    const unsigned ny = (unsigned)std::min(count, 65535);
    const dim3 grid((unsigned)((2LL * cells + 127) / 128), ny);
    fine_resid_kernel<<<grid, 128, 0, (cudaStream_t)stream>>>(B->d_inst, B->d_code, first, count, cells, pred, base,
                                                              V_target, resid, inv, loss);
    CPMDP_CUDA(cudaGetLastError());
    const long long tiles = (long long)zc * ((yc + kGradCells - 1) / kGradCells) * ((xc + kGradCells - 1) / kGradCells);
    fine_grad_kernel<<<dim3((unsigned)tiles, ny), kGradCells * kGradCells, 0, (cudaStream_t)stream>>>(
        B->d_inst, first, count, zc, yc, xc, resid, inv, (__nv_bfloat16 *)dy);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_coarse_vi(const cpmdp_batch *B, int32_t first, int32_t count, float tol, int32_t max_sweeps,
                                float *coarse_v, uint16_t *feat, void *stream) {
    int cells = 0;
    cpmdp_status s = batch_range(B, first, count, &cells);
    if (s != CPMDP_OK) return s;
    if (cells > kMaxCoarseCells) {
        set_error("coarse value iteration holds at most %d coarse cells per instance", kMaxCoarseCells);
        return CPMDP_EINVAL;
    }
    if (!coarse_v || !(tol > 0.f) || max_sweeps < 1) { set_error("coarse_v, tol > 0 and max_sweeps >= 1 required"); return CPMDP_EINVAL; }
    const size_t smem = (size_t)cells * 13;
    const auto kern = cells <= kCoarseThreads ? coarse_vi_kernel<1> : cells <= 4 * kCoarseThreads ? coarse_vi_kernel<4>
                                                                                                  : coarse_vi_kernel<8>;
    CPMDP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<count, kCoarseThreads, smem, (cudaStream_t)stream>>>(B->d_inst, B->d_code, B->d_R, first, cells, tol, max_sweeps,
                                                                coarse_v, (__nv_bfloat16 *)feat);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_conv3d_forward(const uint16_t *x, const uint16_t *wf, const float *bias, uint16_t *y, float *y0,
                                  int32_t n, int32_t z, int32_t yy, int32_t xx, int32_t dilation, int32_t relu,
                                  void *stream) {
    cpmdp_status s = dims_ok(n, z, yy, xx, dilation);
    if (s != CPMDP_OK) return s;
    if (!x || !wf || !y) { set_error("x, w and y are required"); return CPMDP_EINVAL; }
    Dims dm{n, z, yy, xx};
    CPMDP_CUDA(launch_conv((const __nv_bfloat16 *)x, (const uint8_t *)wf, bias, nullptr, (__nv_bfloat16 *)y, y0, dm,
                           dilation, 1, relu, (cudaStream_t)stream));
    return CPMDP_OK;
}

cpmdp_status cpmdp_conv3d_backward_data(const uint16_t *dy, const uint16_t *wb, const uint16_t *act_in, uint16_t *dx,
                                        int32_t n, int32_t z, int32_t yy, int32_t xx, int32_t dilation, void *stream) {
    cpmdp_status s = dims_ok(n, z, yy, xx, dilation);
    if (s != CPMDP_OK) return s;
    if (!dy || !wb || !dx) { set_error("dy, w and dx are required"); return CPMDP_EINVAL; }
    Dims dm{n, z, yy, xx};
    CPMDP_CUDA(launch_conv((const __nv_bfloat16 *)dy, (const uint8_t *)wb, nullptr, (const __nv_bfloat16 *)act_in,
                           (__nv_bfloat16 *)dx, nullptr, dm, dilation, -1, 0, (cudaStream_t)stream));
    return CPMDP_OK;
}

cpmdp_status cpmdp_conv3d_backward_weight(const uint16_t *x, const uint16_t *dy, float *dw, float *db, int32_t n,
                                          int32_t z, int32_t yy, int32_t xx, int32_t dilation, void *stream) {
    cpmdp_status s = dims_ok(n, z, yy, xx, dilation);
    if (s != CPMDP_OK) return s;
    if (!x || !dy || !dw) { set_error("x, dy and dw are required"); return CPMDP_EINVAL; }
    Dims dm{n, z, yy, xx};
    const __nv_bfloat16 *xb = (const __nv_bfloat16 *)x, *db16 = (const __nv_bfloat16 *)dy;
    const cudaError_t e = launch_dw(xb, db16, dw, dm, dilation, (cudaStream_t)stream);
    if (e == cudaErrorNotSupported) {
        const int chunk = 512;
        dim3 grid((dm.nvox() + chunk - 1) / chunk, 27);
        conv_dw_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(xb, db16, dw, dm, dilation, chunk);
        CPMDP_CUDA(cudaGetLastError());
    } else {
        CPMDP_CUDA(e);
    }
    if (db) {
        if (reinterpret_cast<uintptr_t>(dy) & 15)
            conv_db_kernel<<<grid_for(dm.nvox(), 64), 256, 0, (cudaStream_t)stream>>>(db16, db, dm.nvox());
        else
            conv_db_vec_kernel<<<std::min(grid_for(dm.nvox(), 256), 304), 256, 0, (cudaStream_t)stream>>>(
                reinterpret_cast<const uint4 *>(dy), db, dm.nvox());
        CPMDP_CUDA(cudaGetLastError());
    }
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_loss_grad(const float *pred, const float *target, const float *mask, int32_t nvox, uint16_t *dy,
                                float *loss, void *stream) {
    if (nvox < 1 || !pred || !target || !mask || !dy) { set_error("invalid loss arguments"); return CPMDP_EINVAL; }
    loss_grad_kernel<<<grid_for(nvox, 256), 256, 0, (cudaStream_t)stream>>>(pred, target, mask, (__nv_bfloat16 *)dy,
                                                                            loss, nvox);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_adam_step(float *p, const float *g, float *m, float *v, int64_t n, float lr, float beta1,
                             float beta2, float eps, int32_t step, void *stream) {
    if (n < 1 || !p || !g || !m || !v || step < 1) { set_error("invalid Adam arguments"); return CPMDP_EINVAL; }
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, n, lr, beta1, beta2, eps, c1, c2);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_cast_weights(const float *w, uint16_t *wf, uint16_t *wb, int32_t layers, void *stream) {
    if (layers < 1 || !w || !wf || !wb) { set_error("invalid weight-cast arguments"); return CPMDP_EINVAL; }
    const long long n = (long long)layers * 27 * kC * kC;
    cast_weights_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(w, (__nv_bfloat16 *)wf,
                                                                            (__nv_bfloat16 *)wb, n);
    CPMDP_CUDA(cudaGetLastError());
    return CPMDP_OK;
}

cpmdp_status cpmdp_ws_sync(void *stream) {
    CPMDP_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    int e = 0;
    CPMDP_CUDA(cudaMemcpyFromSymbol(&e, g_conv_err, sizeof(int)));
    if (e) {
        const int zero = 0;
        CPMDP_CUDA(cudaMemcpyToSymbol(g_conv_err, &zero, sizeof(int)));
        set_error("a tensor-core wait in a warm-start convolution ran out");
        return CPMDP_ETIMEOUT;
    }
    return CPMDP_OK;
}

}  // extern "C"
