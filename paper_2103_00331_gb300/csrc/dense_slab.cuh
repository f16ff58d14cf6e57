// Fused mode-product chains of the dense CP backup (FP32 / FP64, any shape).
//
// E_a[V] = sum_r lambda_{a,r} (V x_1 U_{a,r,1} ... x_D U_{a,r,D}). The modes
// are cut into runs of consecutive dimensions ("phases", picked by a cost
// model when the model is built). One launch applies one phase of every
// chain (a, r): a block brings a tile of the state tensor to shared memory,
// applies the phase's mode products there one after the other, and stores
// the result; the last phase's blocks own whole rows of states, walk the
// chains, and carry the epilogue (ranks summed in order, Q = R + gamma E,
// max / argmax over actions, residual) in registers. A 4-D sweep is 2
// launches instead of A R D, and a chain's tensor goes through global memory
// once instead of D times.
//
// Tile of a phase that is not the last: for one index of the dimensions
// before it, all G states of its dimensions x w consecutive columns of the
// dimensions after it. Tile of the last phase: g rows (indices of the
// dimensions before it) x all G states. Both pad the innermost line (the
// phase's last dimension with its columns) to an odd number of 16-byte
// granules, so that lanes on neighbouring lines hit different banks. What
// the last phase reads is stored tile by tile ([column tile][G][w]): the
// phase before it writes whole tiles back to back, and g rows of the last
// phase read g w elements at a time. Products run from one of two tile buffers to the other.
// Per thread IB x CB outputs in registers (CB = one 16-byte vector of
// columns); the factor matrix arrives transposed (contraction index first,
// zero-padded) by asynchronous copies, KC contraction steps at a time,
// double-buffered across mode and chain boundaries.
//
// What bounds it: large FP32 models the FMA pipe and the issue slots (the
// first phase of 48 x 50 x 52 x 46, 4 actions, rank 4: half the FMA peak,
// 0.52 ms; the last 1.01 ms), FP64 ones the FP64 pipe (2 multiply-adds per
// cycle and SM), small ones the launches and the latency of a block's chain.
// Measured, one sweep, one launch per mode before / fused now: FP32
// 48 x 50 x 52 x 46 3.08 / 1.54 ms, 64^4 (8 actions, rank 8) 30.2 / 17.4 ms,
// 20^3 (4 actions, rank 3) 0.29 / 0.020 ms; FP64 48 x 50 x 52 x 46 45.3 /
// 32.3 ms, 8^4 (4 actions, rank 3) 1.00 / 0.021 ms.
//
// The arithmetic is the one of mode_product_kernel, in its order: every
// output is one chain of fused multiply-adds over ascending contraction
// index (padding adds exact zeros), so values, policies and residuals are
// the same.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace cpmdp {

enum DenseMode : int { DM_VI = 0, DM_EVAL = 1, DM_IMPROVE = 2, DM_GREEDY = 3, DM_STORE_E = 4 };

constexpr int kSlabThreads = 512;              // largest block (128 registers a thread)
constexpr int kSlabThreadsWide = 384;          // with the wide FP32 tile (168)
constexpr int kSlabSmemMax = 227 * 1024;

// Geometry of one mode of a phase in the tile (see slab_item).
struct SlabMode {
    int N, ni;                 // size, padded factor row
    int Rt;                    // elements from one index of the mode to the next
    int lstr;                  // from one index of the modes before it to the next
    int cols, nib, ncb, per;   // columns (vectors; contiguous dimension: lines), row and column blocks, items
    int uoff;                  // offset of the transposed factor in a chain's block
    float inv_per, inv_r, inv_Rt;
};

// One launch: a phase of a range of chains. Everything a thread needs to find
// its work without dividing is worked out here (inv_x = 1 / x).
struct SlabPhase {
    int nmodes;
    SlabMode m[kMaxDim];
    int G;                     // product of the mode sizes
    int nl, lpr;               // last mode size, lines per row = G / nl
    int w;                     // columns per tile (last phase: rows)
    int wp;                    // columns padded to a vector (last phase: pitch of the last dimension)
    int lp;                    // pitch of a line: the phase's last dimension x wp, padded (last phase: wp)
    int tile;                  // elements of a tile
    int gprev, wprev;          // last phase: G and w of the phase before it (0: X is in state order)
    int ch;                    // chains a block works on at once (last phase), one after the other (the others)
    int kc;                    // contraction steps per factor chunk
    int nimax;                 // largest padded factor row of the phase
    int threads;
    int fine;                  // small register tile
    unsigned smem;
    unsigned ntile;            // column tiles (not the last phase)
    int bufs;                  // tile buffers: 2 when a block works through several chains
    float inv_nl, inv_wprev;
    long long L, Rt;           // states before / after the phase's dimensions
};

struct SlabPlan {
    int nphase = 0;            // 0: no plan fits, mode_product_kernel runs
    SlabPhase ph[kMaxDim];
    long long ublock = 0;      // elements of one chain's transposed factors
    int actions = 0;           // actions per group of launches (what the workspace holds)
    long long chain = 0;       // elements of one chain's intermediate
    size_t ws_bytes = 0;       // intermediates of one group (one buffer; two with 3 phases or more)
};

// The factors of every chain, transposed and padded, the two plans, and the
// workspace of each (one allocation where the first one taken serves both).
struct DenseSlab {
    SlabPlan plan32, plan64;
    float *ut32 = nullptr;
    double *ut64 = nullptr;
    float *lam32 = nullptr;
    double *lam64 = nullptr;
    void *ws32 = nullptr, *ws64 = nullptr;
};

template <typename T>
struct SlabArgs {
    const T *X;                // V (chain stride 0) or the previous phase's output
    T *Y;                      // this phase's output (not the last phase)
    long long xchain, ychain;  // elements between chains of X (0: V) and of Y
    int ytiled;                // Y is stored tile by tile (the last phase reads it)
    const T *ut;
    long long ublock;
    const T *lam;
    int c0, nchains;           // chains of this group
    int rank;
    int a0, a1, nact;          // actions of this group, of the model
    int mode;
    T gamma, margin;
    T *best, *qold;            // per state, between groups of actions / for improvements
    uint8_t *arg;
    const T *R, *Vin;
    T *Vout;
    uint8_t *pi;
    unsigned long long *res;
    unsigned *changed;
    const int *stop;           // nullable: the sweep does nothing when it is set
    SlabPhase p;
};

template <typename T> struct SlabVec;
template <> struct SlabVec<float> { using type = float4; static constexpr int n = 4; };
template <> struct SlabVec<double> { using type = double2; static constexpr int n = 2; };

__device__ __forceinline__ void slab_cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
template <typename T>
__device__ __forceinline__ void slab_cp1(T *dst, const T *src) {
    if (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                     : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                     : "memory");
}
__device__ __forceinline__ void slab_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void slab_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// e / n for 0 <= e < 2^20, n >= 1, with inv = 1 / n: (e + 0.5) / n is at least
// 0.5 / n away from an integer, more than the rounding of the product.
__device__ __forceinline__ int slab_div(int e, float inv) { return __float2int_rd(((float)e + 0.5f) * inv); }

// Largest |a - b| seen so far, as a double. Float values: the exact
// difference of two floats is d + e with d = fl(a - b) and e the rounding
// error (Knuth's two-sum), kept as that pair and widened once at the end, so
// no state costs an FP64 instruction (but for one whose difference is past the
// largest float). NaN differences are skipped, as fmax skips them.
template <typename T> struct SlabMax;
template <> struct SlabMax<double> {
    double m = 0.0;
    __device__ __forceinline__ void add(double a, double b) {
        const double d = fabs(a - b);
        if (d > m) m = d;
    }
    __device__ __forceinline__ double get() const { return m; }
};
template <> struct SlabMax<float> {
    float d = 0.f, e = 0.f;
    double wide = 0.0;         // differences that overflow a float
    __device__ __forceinline__ void add(float a, float b) {
        float s = a - b;
        const float bb = s - a;
        float t = (a - (s - bb)) - (b + bb);
        if (s < 0.f) { s = -s; t = -t; }
        if (s > d || (s == d && t > e)) {
            if (isinf(s)) wide = fmax(wide, fabs((double)a - (double)b));
            else { d = s; e = t; }
        }
    }
    __device__ __forceinline__ double get() const { return fmax(wide, (double)d + (double)e); }
};

// A block's threads split over `nch` chains, and a chain's threads over a
// plane of outer x per units: a thread keeps one column and steps through the
// outer index by a fixed stride, so no loop divides.
struct SlabSplit {
    int k;                     // chain of the group (nch: left over)
    int c, g, dc, dg;          // first column, first outer index, strides
    __device__ __forceinline__ SlabSplit(int nch, int per) {
        const int tpc = slab_div(blockDim.x, __frcp_rn((float)nch));
        k = slab_div(threadIdx.x, __frcp_rn((float)tpc));
        const int t = threadIdx.x - k * tpc;
        dc = min(per, tpc);
        const float inv = __frcp_rn((float)dc);
        dg = slab_div(tpc, inv);
        g = slab_div(t, inv);
        c = t - g * dc;
        if (g >= dg) k = nch;
    }
};

// Factor chunk `k0` of mode q for `nch` chains, into one stage.
template <typename T>
__device__ __forceinline__ void slab_load_u(const SlabArgs<T> &a, int chain, int nch, int q, int k0, T *dst) {
    const SlabMode &m = a.p.m[q];
    const int rows = min(a.p.kc, ((m.N + 3) & ~3) - k0);
    const int vec = 16 / (int)sizeof(T), per = rows * m.ni / vec;
    const T *src = a.ut + chain * a.ublock + (m.uoff + k0 * m.ni);
    if (nch == 1) {
        for (int e = threadIdx.x; e < per; e += blockDim.x) slab_cp16(dst + e * vec, src + e * vec);
        return;
    }
    const SlabSplit sp(nch, per);
    if (sp.k >= nch || sp.g > 0) return;
    src += sp.k * a.ublock;
    T *d = dst + sp.k * a.p.kc * a.p.nimax;
    for (int e = sp.c; e < per; e += sp.dc) slab_cp16(d + e * vec, src + e * vec);
}

// Tile of a phase that is not the last: all G states x w columns from c0 on.
template <typename T>
__device__ __forceinline__ void slab_load_cols(const SlabPhase &p, const T *X, long long l, long long c0, T *dst) {
    constexpr int VW = SlabVec<T>::n;
    const T *src = X + l * p.G * p.Rt + c0;
    const int cols = (int)min((long long)p.w, p.Rt - c0);
    const bool vec = p.Rt % VW == 0 && cols % VW == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    const int step = vec ? VW : 1, nl = p.nl;
    const SlabSplit sp(1, p.wp / step);
    if (sp.k) return;
    const int l0 = slab_div(sp.g, p.inv_nl), i0 = sp.g - l0 * nl, dl = slab_div(sp.dg, p.inv_nl), di = sp.dg - dl * nl;
    for (int c = sp.c; c < p.wp / step; c += sp.dc) {
        const int col = c * step;
        int line = l0, idx = i0;
        const T *s = src + sp.g * p.Rt + col;
        for (int g = sp.g; g < p.G; g += sp.dg) {
            T *d = dst + line * p.lp + idx * p.wp + col;
            if (col >= cols) {
                for (int k = 0; k < step; k++) d[k] = (T)0;
            } else if (vec) {
                slab_cp16(d, s);
            } else {
                slab_cp1(d, s);
            }
            s += sp.dg * p.Rt;
            idx += di;
            line += dl;
            if (idx >= nl) { idx -= nl; line++; }
        }
    }
}

// Tiles of the last phase, one per chain: rows r0 .. r0 + rows - 1, the last
// dimension padded to wp with zeros.
template <typename T>
__device__ __forceinline__ void slab_load_rows(const SlabPhase &p, const T *X, long long xchain, int nch, int r0,
                                               int rows, T *dst) {
    constexpr int VW = SlabVec<T>::n;
    const int nl = p.nl, lines = rows * p.lpr;
    T *const tile0 = dst;
    const bool aligned = nl % VW == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 && xchain % VW == 0;
    if (p.wprev) {
        // stored as tiles of wprev columns: the rows' part of a tile is contiguous
        const int w = p.wprev, tiles = slab_div(p.G + w - 1, p.inv_wprev);
        const bool vec = aligned && w % VW == 0, two = VW == 4 && nl % 2 == 0 && w % 2 == 0 && !vec;
        const int step = vec ? VW : two ? 2 : 1, per = rows * w / step;
        const SlabSplit sp(nch, per);
        if (sp.k < nch) {
            X += sp.k * xchain;
            dst += sp.k * p.tile;
            const int dcg = sp.dg * w, dl = slab_div(dcg, p.inv_nl), di = dcg - dl * nl;
            const long long dsrc = (long long)dcg * p.gprev;
            for (int k = sp.c; k < per; k += sp.dc) {
                const int row = slab_div(k * step, p.inv_wprev), c = k * step - row * w;
                const unsigned R = (unsigned)(r0 + row), lo = R / (unsigned)p.gprev;
                const T *s = X + ((long long)lo * tiles + sp.g) * p.gprev * w + (R - lo * p.gprev) * w + c;
                const int cg0 = sp.g * w + c;
                int li = slab_div(cg0, p.inv_nl), col = cg0 - li * nl;
                T *d0 = dst + row * p.lpr * p.wp;
                for (int cg = cg0; cg < p.G; cg += dcg) {   // the last tile may be narrower
                    T *d = d0 + li * p.wp + col;
                    if (vec) slab_cp16(d, s);
                    else if (two) slab_cp1(reinterpret_cast<double *>(d), reinterpret_cast<const double *>(s));
                    else slab_cp1(d, s);
                    s += dsrc;
                    col += di;
                    li += dl;
                    if (col >= nl) { col -= nl; li++; }
                }
            }
        }
        // the lines' pads
        for (int e = threadIdx.x; e < nch * lines; e += blockDim.x) {
            const int k = slab_div(e, __frcp_rn((float)lines));
            T *d = tile0 + k * p.tile + (e - k * lines) * p.wp;
            for (int j = nl; j < p.wp; j++) d[j] = (T)0;
        }
        return;
    }
    const int step = aligned ? VW : 1;
    const SlabSplit sp(nch, p.wp / step);
    if (sp.k >= nch) return;
    const T *src = X + sp.k * xchain + (long long)r0 * p.G;
    dst += sp.k * p.tile;
    for (int c = sp.c; c < p.wp / step; c += sp.dc) {
        const int col = c * step;
        for (int li = sp.g; li < lines; li += sp.dg) {
            T *d = dst + li * p.wp + col;
            if (col >= nl) {
                for (int k = 0; k < step; k++) d[k] = (T)0;
            } else if (aligned) {
                slab_cp16(d, src + (long long)li * nl + col);
            } else {
                slab_cp1(d, src + (long long)li * nl + col);
            }
        }
    }
}

// NV values of one vector load (NV x sizeof(T) = 8 or 16 bytes).
template <typename T, int NV>
__device__ __forceinline__ void slab_ldn(const T *p, T (&v)[NV]) {
    static_assert(NV * sizeof(T) == 16 || NV * sizeof(T) == 8, "one load");
    if (NV * sizeof(T) == 16) {
        const int4 t = *reinterpret_cast<const int4 *>(p);
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = reinterpret_cast<const T *>(&t)[k];
    } else {
        const int2 t = *reinterpret_cast<const int2 *>(p);
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = reinterpret_cast<const T *>(&t)[k];
    }
}

// IV factor values (16, 8 or 4 bytes).
template <typename T, int IV>
__device__ __forceinline__ void slab_ldu(const T *p, T (&v)[IV]) {
    if constexpr (IV * sizeof(T) >= 8) slab_ldn<T, IV>(p, v);
    else v[0] = p[0];
}

// Pairs of floats in one 64-bit register, and two fused multiply-adds on them.
__device__ __forceinline__ unsigned long long slab_pair(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void slab_unpair(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void slab_fma2(unsigned long long &acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// State s after the last action: its maximum (or its action's value) and argmax.
template <typename T>
__device__ __forceinline__ void slab_finish(const SlabArgs<T> &a, long long s, T best, uint8_t arg, SlabMax<T> &far,
                                            unsigned &chg) {
    if (a.mode == DM_VI || a.mode == DM_EVAL) {
        const T vin = a.Vin[s];
        if (a.Vout) a.Vout[s] = best;
        if (a.pi && a.mode == DM_VI) a.pi[s] = arg;
        far.add(best, vin);
    } else if (a.mode == DM_GREEDY) {
        a.pi[s] = arg;
    } else {   // improve
        const T q0 = a.qold[s];
        const T thr = a.margin * ((T)1 + (q0 < 0 ? -q0 : q0));
        if (a.pi[s] != arg && best > q0 + thr) { a.pi[s] = arg; chg++; }
    }
}

// A thread's place in one mode product: its chain and its IB x CB outputs.
// Output rows i = (ii / IV) nib IV + ib IV + ii % IV (IV = values per factor
// load), output columns: CB / VW vectors (the contiguous dimension: CB
// lines), ncb apart, so that the lanes of a warp read neighbouring granules.
// A tile that is cut short computes the columns it lacks from what the
// buffer holds; they are never stored to global memory.
template <int CV>
struct SlabItem {
    bool on;
    int kch, i0;               // chain of the group, first output row
    int x[CV];                 // offset of each column vector (line) in the tile
    bool ok[CV];
};

template <typename T, int IB, int CB>
__device__ __forceinline__ void slab_item(const SlabPhase &p, const SlabMode &m, bool inner, int nch, SlabItem<CB> &it) {
    constexpr int VW = SlabVec<T>::n, IV = IB < VW ? IB : VW;
    it.on = (int)threadIdx.x < m.per * nch;
    const int t = it.on ? threadIdx.x : 0;
    it.kch = slab_div(t, m.inv_per);
    const int r = t - it.kch * m.per, d = slab_div(r, m.inv_r);
    const int cb = inner ? d : r - d * m.ncb, ib = inner ? r - d * m.nib : d;
    it.i0 = ib * IV;
#pragma unroll
    for (int b = 0; b < CB; b++) {
        if (b >= (inner ? CB : CB / VW)) break;
        const int c = cb + b * m.ncb, cc = min(c, m.cols - 1);
        it.ok[b] = it.on && c < m.cols;
        const int li = inner ? cc : slab_div(cc * VW, m.inv_Rt);
        it.x[b] = inner ? cc * p.wp : li * m.lstr + cc * VW - li * m.Rt;
    }
}

// The phase. LAST: the phase with the epilogue. NM: 2 for phases of one or
// two modes (the items' places are kept in registers), 0 for more.
template <typename T, int IB, int CB, bool LAST, int NM>
__global__ void __maxnreg__(IB * CB == 64 ? 168 : 128) slab_kernel(const __grid_constant__ SlabArgs<T> a) {
    constexpr int VW = SlabVec<T>::n, IV = IB < VW ? IB : VW;
    constexpr int KS = IB * CB;                // outputs per thread
    constexpr int XV = KS == 64 ? 2 : VW;      // contraction steps per load of a line
    extern __shared__ __align__(16) unsigned char slab_raw[];
    const SlabPhase &p = a.p;
    const int tid = threadIdx.x;
    const unsigned l = LAST ? 0 : blockIdx.x / p.ntile, ct = blockIdx.x - l * p.ntile;
    const long long c0 = LAST ? 0 : (long long)ct * p.w;
    const int r0 = LAST ? blockIdx.x * p.w : 0;
    const int rows = LAST ? min(p.w, (int)p.L - r0) : 1;
    const int nlast = p.nl, tilemax = p.tile;
    const int chmax = LAST ? p.ch : 1;
    // Two tiles when the block works through several (groups of) chains. The
    // next chain's tile arrives in the other one while this chain's products
    // run; in the first phase, where every chain reads the same input, one
    // keeps that input and the first mode writes to the other.
    T *tile = reinterpret_cast<T *>(slab_raw);
    const int other = (p.bufs - 1) * chmax * tilemax;
    T *us = tile + (size_t)p.bufs * chmax * tilemax;
    const int ustage = chmax * p.kc * p.nimax;

    // Who keeps a state's sum over ranks and running maximum. Up to 8 states a
    // thread: registers, states tid + m blockDim. More (the wide FP32 tile):
    // the sum stays with the item's outputs and passes through the tile
    // once per action; the maximum is kept in global memory.
    constexpr bool kOwn = LAST && KS > 8;
    T E[LAST ? KS : 1], best[LAST && !kOwn ? KS : 1];
    uint32_t arg[LAST && !kOwn ? (KS + 3) / 4 : 1];
    SlabMax<T> far;
    unsigned chg = 0;
    const int nstates = rows * p.G;
    const long long S = p.L * p.G * p.Rt;
    int stage = 0;
    const int first = LAST ? 0 : (int)blockIdx.y * p.ch;
    const int nchains = LAST ? a.nchains : min(p.ch, a.nchains - first);

    SlabItem<CB> items[NM > 0 ? NM : 1];
    if (NM > 0) {
#pragma unroll
        for (int q = 0; q < NM; q++)
            if (q < p.nmodes) slab_item<T, IB, CB>(p, p.m[q], LAST && q == p.nmodes - 1, chmax, items[NM > 0 ? q : 0]);
    }

    auto load_tile = [&](int c, int nch, T *dst) {
        const T *X = a.X + (first + c) * a.xchain;
        if (LAST) slab_load_rows<T>(p, X, a.xchain, nch, r0, rows, dst);
        else slab_load_cols<T>(p, X, l, c0, dst);
    };

    // One mode product from src to dst, which may be one tile: all outputs are
    // in registers before the first of them is written. The wide FP32 tile
    // multiplies pairs of output rows with one packed instruction (two
    // independent fused multiply-adds): half the instructions to issue.
    constexpr bool kPack = sizeof(T) == 4 && IB == 8;
    auto mode = [&](const SlabItem<CB> &it, int q, int c, int nch, const T *src, T *dst, bool prefetch) {
        T acc[IB][CB];
        unsigned long long acc2[kPack ? IB / 2 : 1][kPack ? CB : 1];
        if (kPack) {
#pragma unroll
            for (int i = 0; i < (kPack ? IB / 2 : 1); i++)
#pragma unroll
                for (int b = 0; b < (kPack ? CB : 1); b++) acc2[i][b] = 0ull;
        } else {
#pragma unroll
            for (int i = 0; i < IB; i++)
#pragma unroll
                for (int b = 0; b < CB; b++) acc[i][b] = (T)0;
        }
        const SlabMode &m = p.m[q];
        const bool inner = LAST && q == p.nmodes - 1;   // the contiguous dimension
        const bool on = it.on && it.kch < nch;
        const T *in = src + (size_t)it.kch * tilemax;
        T *out = dst + (size_t)it.kch * tilemax;
        // one contraction step: CB inputs, IB factor values
        auto step = [&](const T (&x)[CB], const T *u, int ug) {
            T uu[IB];
#pragma unroll
            for (int g = 0; g < IB / IV; g++) {
                T t[IV];
                slab_ldu<T, IV>(u + g * ug, t);
#pragma unroll
                for (int i = 0; i < IV; i++) uu[g * IV + i] = t[i];
            }
            if constexpr (kPack) {
                unsigned long long u2[IB / 2];
#pragma unroll
                for (int i = 0; i < IB / 2; i++) u2[i] = slab_pair(uu[2 * i], uu[2 * i + 1]);
#pragma unroll
                for (int b = 0; b < CB; b++) {
                    const unsigned long long x2 = slab_pair(x[b], x[b]);
#pragma unroll
                    for (int i = 0; i < IB / 2; i++) slab_fma2(acc2[i][b], u2[i], x2);
                }
            } else {
#pragma unroll
                for (int i = 0; i < IB; i++)
#pragma unroll
                    for (int b = 0; b < CB; b++) acc[i][b] = fma(uu[i], x[b], acc[i][b]);
            }
        };
        for (int k0 = 0; k0 < m.N; k0 += p.kc) {
            slab_wait_all();
            __syncthreads();   // this chunk (and the tile) landed; the other stage is free
            {
                int nq = q, nk = k0 + p.kc, nc = c, nn = nch;
                if (nk >= m.N) {
                    nk = 0;
                    if (++nq == p.nmodes) { nq = 0; nc = c + chmax; nn = min(chmax, nchains - nc); }
                }
                if (nc < nchains) slab_load_u<T>(a, a.c0 + first + nc, nn, nq, nk, us + (stage ^ 1) * ustage);
                if (prefetch && k0 == 0) load_tile(c + chmax, min(chmax, nchains - c - chmax), dst == tile ? tile + other : tile);
                slab_commit();
            }
            if (on) {
                const T *u = us + stage * ustage + it.kch * p.kc * p.nimax + it.i0;
                const int kn = min(p.kc, m.N - k0), ni = m.ni, ug = m.nib * IV;
                if (inner) {
                    const T *xp = in + k0;
                    for (int j = 0; j < kn; j += XV) {     // rows of U past N are zero, so are the pads of x
                        T x[CB][XV];
#pragma unroll
                        for (int b = 0; b < CB; b++) slab_ldn<T, XV>(xp + it.x[b] + j, x[b]);
#pragma unroll
                        for (int v = 0; v < XV; v++) {
                            T xv[CB];
#pragma unroll
                            for (int b = 0; b < CB; b++) xv[b] = x[b][v];
                            step(xv, u, ug);
                            u += ni;
                        }
                    }
                } else {
                    const T *xp[CB / VW];
#pragma unroll
                    for (int b = 0; b < CB / VW; b++) xp[b] = in + it.x[b] + k0 * m.Rt;
                    const int rt = m.Rt;
#pragma unroll 4
                    for (int j = 0; j < kn; j++) {
                        T x[CB];
#pragma unroll
                        for (int b = 0; b < CB / VW; b++) {
                            T t[VW];
                            slab_ldn<T, VW>(xp[b], t);
                            xp[b] += rt;
#pragma unroll
                            for (int v = 0; v < VW; v++) x[b * VW + v] = t[v];
                        }
                        step(x, u, ug);
                        u += ni;
                    }
                }
            }
            stage ^= 1;
        }
        if constexpr (kPack) {
#pragma unroll
            for (int i = 0; i < IB / 2; i++)
#pragma unroll
                for (int b = 0; b < CB; b++) slab_unpair(acc2[i][b], acc[2 * i][b], acc[2 * i + 1][b]);
        }
        if (kOwn && inner) {
            const int chain = a.c0 + c, r = chain % a.rank;
            const T lam = a.lam[chain];
#pragma unroll
            for (int i = 0; i < IB; i++)
#pragma unroll
                for (int b = 0; b < CB; b++) {
                    E[LAST ? i * CB + b : 0] = fma(lam, acc[i][b], r == 0 ? (T)0 : E[LAST ? i * CB + b : 0]);
                    acc[i][b] = E[LAST ? i * CB + b : 0];
                }
        }
        if (src == dst) __syncthreads();   // every input of this mode was read
        // the sums of ranks are stored once an action is complete
        if (!on || (kOwn && inner && (a.c0 + c + 1) % a.rank != 0)) return;
#pragma unroll
        for (int g = 0; g < IB / IV; g++) {
            const int i0 = it.i0 + g * m.nib * IV;
            if (inner) {
#pragma unroll
                for (int b = 0; b < CB; b++) {
                    if (!it.ok[b]) continue;
                    T *o = out + it.x[b] + i0;
                    if (IV == VW) {
                        typename SlabVec<T>::type v;
#pragma unroll
                        for (int k = 0; k < IV; k++) reinterpret_cast<T *>(&v)[k] = acc[g * IV + k][b];
                        if (i0 < m.N) *reinterpret_cast<typename SlabVec<T>::type *>(o) = v;   // may run into the line's pads
                    } else {
#pragma unroll
                        for (int k = 0; k < IV; k++)
                            if (i0 + k < m.N) o[k] = acc[g * IV + k][b];
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < IV; k++) {
                    if (i0 + k >= m.N) continue;
#pragma unroll
                    for (int b = 0; b < CB / VW; b++) {
                        if (!it.ok[b]) continue;
                        typename SlabVec<T>::type v;
#pragma unroll
                        for (int e = 0; e < VW; e++) reinterpret_cast<T *>(&v)[e] = acc[g * IV + k][b * VW + e];
                        *reinterpret_cast<typename SlabVec<T>::type *>(out + it.x[b] + (i0 + k) * m.Rt) = v;
                    }
                }
            }
        }
    };

    slab_load_u<T>(a, a.c0 + first, min(chmax, nchains), 0, 0, us);
    load_tile(0, min(chmax, nchains), tile);
    slab_commit();
    if (a.stop) {
        // read while the first copies fly; the same for every thread
        const int stopped = *a.stop;
        slab_wait_all();
        if (stopped) return;
    }
    for (int c = 0; c < nchains; c += chmax) {
        const int nch = min(chmax, nchains - c);
        // this chain's products run in `work`
        const bool keep = !LAST && a.xchain == 0;
        const int turn = LAST ? c / chmax : c;
        T *work = keep ? tile + other : tile + (turn & 1) * other;
        const bool prefetch = !keep && c + chmax < nchains;
        if (NM > 0) {
#pragma unroll
            for (int q = 0; q < NM; q++)
                if (q < p.nmodes) mode(items[NM > 0 ? q : 0], q, c, nch, keep && q == 0 ? tile : work, work, prefetch && q == 0);
        } else {
            for (int q = 0; q < p.nmodes; q++) {
                SlabItem<CB> it;
                slab_item<T, IB, CB>(p, p.m[q], LAST && q == p.nmodes - 1, chmax, it);
                mode(it, q, c, nch, keep && q == 0 ? tile : work, work, prefetch && q == 0);
            }
        }
        if (!LAST) {
            // store the tile
            __syncthreads();
            T *dst = a.Y + (long long)(first + c) * a.ychain;
            const int cols = (int)min((long long)p.w, p.Rt - c0);
            long long pitch = p.Rt;
            if (a.ytiled) {
                dst += ((long long)l * p.ntile + ct) * p.G * p.w;
                pitch = p.w;
            } else {
                dst += (long long)l * p.G * p.Rt + c0;
            }
            const bool vec = pitch % VW == 0 && cols % VW == 0;
            const int step = vec ? VW : 1;
            const SlabSplit sp(1, cols / step);
            const int l0 = slab_div(sp.g, p.inv_nl), i0 = sp.g - l0 * nlast;
            const int dl = slab_div(sp.dg, p.inv_nl), di = sp.dg - dl * nlast;
            for (int cc = sp.k ? cols : sp.c; cc < cols / step; cc += sp.dc) {
                int line = l0, idx = i0;
                T *d = dst + sp.g * pitch + cc * step;
                for (int g = sp.g; g < p.G; g += sp.dg) {
                    const T *s = work + line * p.lp + idx * p.wp + cc * step;
                    if (vec) *reinterpret_cast<int4 *>(d) = *reinterpret_cast<const int4 *>(s);
                    else *d = *s;
                    d += sp.dg * pitch;
                    idx += di;
                    line += dl;
                    if (idx >= nlast) { idx -= nlast; line++; }
                }
            }
            if (c + chmax < nchains) __syncthreads();   // the tile is free again
        } else if (kOwn) {
            const int chain = a.c0 + c, act = chain / a.rank;
            const bool first_act = act == 0, last_act = act == a.nact - 1;
            if (chain - act * a.rank == a.rank - 1) {
                __syncthreads();
#pragma unroll 4
                for (int st = tid; st < nstates; st += blockDim.x) {
                    const int li = slab_div(st, p.inv_nl);
                    const T e = work[li * p.wp + st - li * nlast];
                    const long long s = (long long)r0 * p.G + st;
                    if (a.mode == DM_STORE_E) {
                        // E_a in the tensor-core pass-B layout (64^4): [a][(i3,i4)][(i1,i2)]
                        a.Vout[(long long)act * S + (s % 4096) * 4096 + s / 4096] = e;
                        continue;
                    }
                    const T qv = fma(a.gamma, e, a.R[s]);
                    T b0 = first_act ? qv : a.best[s];
                    uint8_t ar = 0;
                    if (a.mode == DM_EVAL) {
                        if (a.pi[s] == act) b0 = qv;
                    } else if (!first_act) {
                        ar = a.arg[s];
                        if (qv > b0) { b0 = qv; ar = (uint8_t)act; }
                    }
                    if (a.mode == DM_IMPROVE && a.pi[s] == act) a.qold[s] = qv;
                    if (last_act) {
                        slab_finish<T>(a, s, b0, ar, far, chg);
                    } else {
                        a.best[s] = b0;
                        if (a.mode != DM_EVAL) a.arg[s] = ar;
                    }
                }
                __syncthreads();   // the tile is free again
            }
        } else {
            __syncthreads();
            for (int k = 0; k < nch; k++) {
                const int chain = a.c0 + c + k, act = chain / a.rank, r = chain - act * a.rank;
                const T lam = a.lam[chain];
                const T *in = work + (size_t)k * tilemax;
                const bool last_rank = r == a.rank - 1, first_act = act == 0, last_act = act == a.nact - 1;
#pragma unroll
                for (int m = 0; m < (kOwn ? 0 : KS); m++) {
                    const int st = tid + m * (int)blockDim.x;
                    if (st >= nstates) continue;
                    const int li = slab_div(st, p.inv_nl);
                    const T e = fma(lam, in[li * p.wp + st - li * nlast], r == 0 ? (T)0 : E[m]);
                    E[m] = e;
                    if (!last_rank) continue;
                    const long long s = (long long)r0 * p.G + st;
                    if (a.mode == DM_STORE_E) {
                        a.Vout[(long long)act * S + (s % 4096) * 4096 + s / 4096] = e;
                        continue;
                    }
                    const T qv = fma(a.gamma, e, a.R[s]);
                    const int sh = 8 * (m & 3);
                    const bool resumed = act == a.a0 && !first_act;   // this group of launches starts here
                    T b0 = resumed ? a.best[s] : best[m];
                    if (a.mode == DM_EVAL) {
                        if (first_act || a.pi[s] == act) b0 = qv;
                    } else {
                        if (resumed) arg[m / 4] = (arg[m / 4] & ~(0xFFu << sh)) | ((uint32_t)a.arg[s] << sh);
                        if (first_act || qv > b0) {
                            b0 = qv;
                            arg[m / 4] = (arg[m / 4] & ~(0xFFu << sh)) | ((uint32_t)act << sh);
                        }
                    }
                    best[m] = b0;
                    if (a.mode == DM_IMPROVE && a.pi[s] == act) a.qold[s] = qv;
                    if (act == a.a1 - 1 && !last_act) {
                        a.best[s] = b0;
                        if (a.mode != DM_EVAL) a.arg[s] = (uint8_t)(arg[m / 4] >> sh);
                    }
                }
            }
            if (c + chmax < nchains) __syncthreads();   // the tiles are free again
        }
    }
    if (LAST && a.a1 == a.nact && a.mode != DM_STORE_E) {
        if (!kOwn) {
#pragma unroll
            for (int m = 0; m < (kOwn ? 0 : KS); m++) {
                const int st = tid + m * (int)blockDim.x;
                if (st < nstates)
                    slab_finish<T>(a, (long long)r0 * p.G + st, best[m], (uint8_t)(arg[m / 4] >> (8 * (m & 3))), far, chg);
            }
        }
        if (a.res) {
            // non-negative doubles order like their bits (no NaN among them)
            const unsigned long long bits = (unsigned long long)__double_as_longlong(far.get());
            const unsigned hi = (unsigned)(bits >> 32), hm = __reduce_max_sync(0xFFFFFFFFu, hi);
            const unsigned lm = __reduce_max_sync(0xFFFFFFFFu, hi == hm ? (unsigned)bits : 0u);
            if ((tid & 31) == 0 && (hm | lm)) atomicMax(a.res, ((unsigned long long)hm << 32) | lm);
        }
        if (a.changed) {
            const unsigned n = __reduce_add_sync(0xFFFFFFFFu, chg);
            if ((tid & 31) == 0 && n) atomicAdd(a.changed, n);
        }
    }
}

// Build the plans and the transposed factors (model build). A model without a
// plan, or without the memory for its factors, has nphase == 0.
cpmdp_status slab_prepare(Factors &F);
// The workspace of sweeps of `elem`-byte values; without the memory for it the plan is dropped.
void slab_workspace(const Factors &F, size_t elem);
void slab_free(Factors &F);
const SlabPlan *slab_plan(const Factors &F, size_t elem);

// One sweep over all chains (see dense_sweep for the modes).
template <typename T>
cudaError_t slab_sweep(const Factors &F, const T *Vin, T *Vout, uint8_t *pi, int mode, T margin,
                       unsigned long long *res, unsigned *chg, const int *stop, cudaStream_t st);

}  // namespace cpmdp
