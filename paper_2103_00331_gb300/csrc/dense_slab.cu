// Plans, workspace and launches of the fused mode-product chains
// (dense_slab.cuh).
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "dense_slab.cuh"

namespace cpmdp {

// ut[k][i] = U[i][k], zero-padded to n4 x ni, for every chain (blockIdx.y) and mode.
struct UtGeom {
    int ndim;
    int N[kMaxDim];
    int src[kMaxDim], dst[kMaxDim];
    long long sblock, dblock;
};

template <typename T>
__global__ void slab_transpose_kernel(const double *__restrict__ U, T *__restrict__ ut, UtGeom g) {
    const double *u = U + (long long)blockIdx.y * g.sblock;
    T *o = ut + (long long)blockIdx.y * g.dblock;
    for (int d = 0; d < g.ndim; d++) {
        const int n = g.N[d], ni = (n + 7) & ~7, n4 = (n + 3) & ~3;
        for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n4 * ni;
             e += (long long)gridDim.x * blockDim.x) {
            const int k = (int)(e / ni), i = (int)(e % ni);
            o[g.dst[d] + e] = k < n && i < n ? (T)u[g.src[d] + (long long)i * n + k] : (T)0;
        }
    }
}

// ---------------------------------------------------------------------------
// planning

struct PhaseCost {
    SlabPhase ph;
    double cycles;
    bool ok;
};

// Best tile of the phase [d0, d1) and its estimated cycles. The estimate
// follows a block: copies (a latency), then per mode the larger of its
// threads' own instruction chain and the SM's multiply-add rate over the
// blocks it holds; blocks run in waves. FP64 runs at 2 multiply-adds per
// cycle and SM on GB300, and a warp can use a quarter of that, so small FP64
// tiles want many warps of few outputs.
template <typename T>
static PhaseCost plan_phase(const Factors &F, int d0, int d1, int nchains, const int *uoff) {
    constexpr int VW = (int)(16 / sizeof(T));
    constexpr bool f64 = sizeof(T) == 8;
    const bool last = d1 == F.ndim;
    PhaseCost best;
    memset(&best, 0, sizeof(best));
    SlabPhase p;
    memset(&p, 0, sizeof(p));
    p.nmodes = d1 - d0;
    long long G = 1, L = 1, Rt = 1;
    for (int d = 0; d < d0; d++) L *= F.shape[d];
    for (int d = d1; d < F.ndim; d++) Rt *= F.shape[d];
    for (int d = d0; d < d1; d++) {
        G *= F.shape[d];
        if (G > (1 << 16)) return best;
        p.m[d - d0].N = (int)F.shape[d];
        p.m[d - d0].ni = ((int)F.shape[d] + 7) & ~7;
        p.m[d - d0].uoff = uoff[d];
        p.nimax = std::max(p.nimax, ((int)F.shape[d] + 7) & ~7);
    }
    p.G = (int)G;
    p.L = L;
    p.Rt = Rt;
    const int nl = p.m[p.nmodes - 1].N;
    p.nl = nl;
    p.lpr = (int)(G / nl);
    p.inv_nl = 1.f / (float)nl;
    const double sms = std::max(1, F.num_sms);
    for (int fine = 0; fine < 2; fine++) {
        const int IB = fine ? (f64 ? 1 : 2) : (f64 ? 4 : 8), CB = !fine && !f64 && !last ? 8 : VW;
        // the wide FP32 tile keeps one chain's sums in its items' registers
        const int chmost = last && (f64 || fine) ? std::min(nchains, 64) : 1;
        for (int ch = 1; ch <= (last ? chmost : std::min(nchains, 16)); ch++) {
            if (ch > 1 && nchains % ch) continue;
            for (long long w = last ? 1 : std::min<long long>(VW, Rt);; w *= 2) {
                if (w > (last ? L : ((Rt + VW - 1) / VW) * VW) && w > 1 && w / 2 >= (last ? L : Rt)) break;
                p.fine = fine;
                p.ch = ch;
                p.w = (int)std::min<long long>(w, last ? L : Rt);
                if (last) {
                    p.wp = ((nl + VW - 1) / VW) * VW;
                    if ((p.wp / VW) % 2 == 0) p.wp += VW;   // odd 16-byte granules: neighbouring lines, other banks
                } else {
                    p.wp = ((p.w + VW - 1) / VW) * VW;
                }
                p.lp = last ? p.wp : nl * p.wp;
                if ((p.lp / VW) % 2 == 0) p.lp += VW;
                const long long lines = (last ? p.w : 1) * (G / nl);
                if (lines * p.lp > 60000) break;
                long long items = 0;
                double fma = 0, chain = 0, busy = 4;
                p.tile = (int)(lines * p.lp);
                for (int q = p.nmodes - 1, Rq = 0; q >= 0; q--) {
                    SlabMode &m = p.m[q];
                    const int N = m.N;
                    const bool tail = q == p.nmodes - 1, inner = last && tail;
                    Rq = tail ? p.wp : q == p.nmodes - 2 ? p.lp : Rq * p.m[q + 1].N;
                    m.Rt = inner ? 1 : Rq;
                    m.lstr = tail ? p.lp : N * Rq;
                    m.cols = (int)(inner ? lines : (tail ? lines * p.wp : lines / N * p.lp) / VW);
                    const int nc = inner ? CB : CB / VW;
                    m.nib = (N + IB - 1) / IB;
                    m.ncb = (m.cols + nc - 1) / nc;
                    m.per = m.nib * m.ncb;
                    m.inv_per = 1.f / (float)m.per;
                    m.inv_r = 1.f / (float)(inner ? m.nib : m.ncb);
                    m.inv_Rt = 1.f / (float)m.Rt;
                    const long long it = (long long)m.per * (last ? ch : 1);
                    items = std::max(items, it);
                    const double warps = (double)((it + 31) / 32);
                    busy = std::min(busy, warps);
                    fma += warps * 32 * IB * CB * N;
                    // one warp's own pace: FP64 a quarter of the SM's rate, loads and issue otherwise
                    chain += 400 + N * (f64 ? IB * CB * 64.0 + 10 : IB * CB + 14.0);
                }
                if (items > (IB * CB < 64 ? kSlabThreads : kSlabThreadsWide)) break;
                p.threads = (int)std::max<long long>(32, (items + 31) / 32 * 32);
                int nmax = 0;
                for (int q = 0; q < p.nmodes; q++) nmax = std::max(nmax, (p.m[q].N + 3) & ~3);
                p.bufs = last ? (ch < nchains ? 2 : 1) : (ch > 1 ? 2 : 1);
                const size_t tiles = (size_t)p.bufs * (last ? ch : 1) * (size_t)(lines * p.lp) * sizeof(T);
                const size_t urow = 2 * (size_t)(last ? ch : 1) * p.nimax * sizeof(T);
                // registers are a quarter of the SM's per scheduler
                const int regs = IB * CB == 64 ? 168 : last ? 128 : 96;
                double occ = std::min(std::floor(2048.0 / p.threads),
                                      std::floor(4 * std::floor(16384.0 / (regs * 32)) / (p.threads / 32)));
                // the longest factor chunks (fewest barriers) that leave shared memory for those blocks
                auto fit = [&](int kc) { return std::floor(227.0 * 1024 / (tiles + urow * (double)kc + 1024.0)); };
                int kc = std::min(nmax, 64);
                while (kc > 16 && fit(kc) < occ) kc = std::max(16, (kc / 2 + 3) & ~3);
                while (kc > 4 && fit(kc) < 1) kc = std::max(4, (kc / 2) & ~3);
                p.kc = kc;
                p.smem = (unsigned)(tiles + urow * kc);
                if (p.smem > (unsigned)kSlabSmemMax) break;
                occ = std::max(1.0, std::min(occ, fit(kc)));
                const double tiles_x = last ? std::ceil((double)L / p.w) : (double)L * std::ceil((double)Rt / p.w);
                p.ntile = last ? 0u : (unsigned)((Rt + p.w - 1) / p.w);
                const double blocks = last ? tiles_x : tiles_x * std::ceil((double)nchains / ch);
                const double passes = last ? std::ceil((double)nchains / ch) : ch;
                const double here = std::min(occ, std::ceil(blocks / sms));
                const double rate = f64 ? 2.0 * std::min(4.0, busy * here) / 4.0 : 70.0;
                const double pass = 1500 + std::max(chain, here * fma / rate) +
                                    (last ? (double)ch * 30 * std::ceil((double)(p.w * G) / p.threads) : 200.0);
                // tensors in and out, at about HBM rate
                const double mem = (double)nchains * F.nstates * sizeof(T) * ((d0 > 0 ? 1.0 : 0.2) + (last ? 0.0 : 1.0)) / 3000.0;
                const double cyc = 4000 + std::ceil(blocks / (sms * here)) * (passes * pass + 800) + mem;
                if (!best.ok || cyc < best.cycles) {
                    best.ok = true;
                    best.cycles = cyc;
                    best.ph = p;
                }
                if (p.w >= (last ? L : Rt)) break;
            }
        }
    }
    return best;
}

// Whether one launch per mode is faster than the plan. A block of a phase reads
// every factor of the phase whole, which a single SM does at about 50 GB/s (FP32;
// FP64: the SM's multiply-adds); a mode-product launch splits a long mode's rows
// over many blocks, and takes 0.11 us per contraction step (FP64 1.07), up to
// 1.75 times that where the factors outgrow the L2. So modes of more than 1,024
// states lose where one wave of blocks walks few chains. Measured, fused / one
// launch per mode, FP32: 1,500 states 223 / 172 us with one chain, 385 / 333 with
// two, 2,209 / 3,471 with twelve; 2,000 states 613 / 435 with two; 2,500 x 4 780
// / 563 with two; 1,500 x 32 316 / 365 with two. FP64: 2,000 states 4,706 / 4,238
// with two, 1,500 states 2,614 / 3,194.
template <typename T>
static bool modes_faster(const Factors &F, const SlabPlan &plan) {
    constexpr bool f64 = sizeof(T) == 8;
    const double chains = (double)F.nactions * F.rank, sms = F.num_sms;
    double fused = 0, modes = 0, bytes = 0;
    bool longer = false;
    for (int d = 0; d < F.ndim; d++) {
        const double n = (double)F.shape[d];
        longer |= n > 1024;
        modes += chains * std::max(3.0, (f64 ? 1.07 : 0.11) * n);
        bytes += chains * n * n * sizeof(T);
    }
    if (!longer) return false;
    if (!f64) modes *= std::min(1.75, std::max(1.0, bytes / (64 << 20)));
    for (int i = 0; i < plan.nphase; i++) {
        const SlabPhase &p = plan.ph[i];
        const bool last = i == plan.nphase - 1;
        const double blocks = last ? std::ceil((double)p.L / p.w) : (double)p.L * p.ntile * std::ceil(chains / p.ch);
        const double passes = (last ? std::ceil(chains / p.ch) : p.ch) * std::ceil(blocks / sms);
        double factor = 0;
        for (int q = 0; q < p.nmodes; q++) {
            if (last && blocks > sms && p.m[q].N > 1024) return false;
            factor += (double)p.m[q].N * p.m[q].N;
        }
        fused += f64 ? 5.9e-4 * factor * passes : last ? 50 + 7.8e-5 * factor * passes : 1.25e-4 * factor * passes;
    }
    return fused > modes;
}

template <typename T>
static void make_plan(const Factors &F, SlabPlan &plan) {
    const int D = F.ndim;
    const long long nchains_all = (long long)F.nactions * F.rank;
    plan.nphase = 0;
    if (nchains_all > 65535 || F.num_sms < 1) return;
    int uoff[kMaxDim];
    long long off = 0;
    for (int d = 0; d < D; d++) {
        const long long n = F.shape[d];
        uoff[d] = (int)off;
        off += ((n + 3) & ~3LL) * ((n + 7) & ~7LL);
    }
    if (off > (1LL << 28)) return;
    plan.ublock = off;
    // Intermediates of whole actions per group of launches: all of them up to
    // 1 GiB a buffer, at least one action.
    auto groups = [&](long long chain) {
        const double per = (double)F.rank * (double)chain * sizeof(T);
        return (int)std::max(1.0, std::min((double)F.nactions, std::floor((double)(1u << 30) / per)));
    };
    plan.actions = groups(F.nstates);
    const int nch = plan.actions * F.rank;
    // cheapest cut of the dimensions into phases
    double cost[kMaxDim + 1];
    int from[kMaxDim + 1];
    PhaseCost step[kMaxDim + 1];
    cost[0] = 0;
    for (int d1 = 1; d1 <= D; d1++) {
        cost[d1] = -1;
        for (int d0 = 0; d0 < d1; d0++) {
            if (cost[d0] < 0) continue;
            const PhaseCost c = plan_phase<T>(F, d0, d1, nch, uoff);
            if (!c.ok) continue;
            if (cost[d1] < 0 || cost[d0] + c.cycles < cost[d1]) {
                cost[d1] = cost[d0] + c.cycles;
                from[d1] = d0;
                step[d1] = c;
            }
        }
    }
    if (cost[D] < 0) return;
    int cuts[kMaxDim + 1], n = 0;
    for (int d = D; d > 0; d = from[d]) cuts[n++] = d;
    plan.nphase = n;
    for (int i = 0; i < n; i++) plan.ph[i] = step[cuts[n - 1 - i]].ph;
    plan.chain = F.nstates;
    if (n > 1) {
        SlabPhase &z = plan.ph[n - 1], &y = plan.ph[n - 2];
        z.gprev = y.G;
        z.wprev = y.w;
        z.inv_wprev = 1.f / (float)y.w;
        plan.chain = y.L * ((y.Rt + y.w - 1) / y.w) * y.w * y.G;   // whole tiles
        plan.chain = (std::max<long long>(plan.chain, F.nstates) + 3) & ~3LL;
        plan.actions = groups(plan.chain);
    }
    plan.ws_bytes = n > 1 ? (size_t)(n > 2 ? 2 : 1) * (size_t)plan.actions * F.rank * (size_t)plan.chain * sizeof(T) : 0;
    if (modes_faster<T>(F, plan)) plan.nphase = 0;
}

template <typename T>
static cudaError_t slab_attr() {
    constexpr int kWide = sizeof(T) == 8 ? 4 : 8, kWideC = sizeof(T) == 8 ? 2 : 8, kWideL = sizeof(T) == 8 ? 2 : 4;
    constexpr int kFine = sizeof(T) == 8 ? 1 : 2, kFineC = sizeof(T) == 8 ? 2 : 4;
    const void *k[] = {(const void *)slab_kernel<T, kWide, kWideC, false, 0>, (const void *)slab_kernel<T, kWide, kWideL, true, 0>,
                       (const void *)slab_kernel<T, kWide, kWideC, false, 2>, (const void *)slab_kernel<T, kWide, kWideL, true, 2>,
                       (const void *)slab_kernel<T, kFine, kFineC, false, 0>, (const void *)slab_kernel<T, kFine, kFineC, true, 0>,
                       (const void *)slab_kernel<T, kFine, kFineC, false, 2>, (const void *)slab_kernel<T, kFine, kFineC, true, 2>};
    for (const void *f : k) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSlabSmemMax);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void slab_free(Factors &F) {
    if (!F.slab) return;
    cudaFree(F.slab->ut32);
    cudaFree(F.slab->ut64);
    cudaFree(F.slab->lam32);
    cudaFree(F.slab->lam64);
    cudaFree(F.slab->ws32);
    if (F.slab->ws64 != F.slab->ws32) cudaFree(F.slab->ws64);
    delete F.slab;
    F.slab = nullptr;
}

cpmdp_status slab_prepare(Factors &F) {
    DenseSlab *s = new (std::nothrow) DenseSlab;
    if (!s) { set_error("out of host memory"); return CPMDP_ENOMEM; }
    F.slab = s;
    make_plan<float>(F, s->plan32);
    make_plan<double>(F, s->plan64);
    const size_t nch = (size_t)F.nactions * F.rank;
    std::vector<float> l32(nch);
    for (size_t i = 0; i < nch; i++) l32[i] = (float)F.lambda[i];
    CPMDP_CUDA(slab_attr<float>());
    CPMDP_CUDA(slab_attr<double>());
    UtGeom g;
    memset(&g, 0, sizeof(g));
    g.ndim = F.ndim;
    long long so = 0, dof = 0;
    for (int d = 0; d < F.ndim; d++) {
        const long long n = F.shape[d];
        g.N[d] = (int)n;
        g.src[d] = (int)so;
        g.dst[d] = (int)dof;
        so += n * n;
        dof += ((n + 3) & ~3LL) * ((n + 7) & ~7LL);
    }
    g.sblock = so;
    g.dblock = dof;
    // A plan is an option: without the memory for its factors it is dropped.
    const dim3 grid(16, (unsigned)nch);
    auto put = [&](SlabPlan &plan, auto *&ut, auto *&lam, const void *host) -> cudaError_t {
        typedef typename std::remove_reference<decltype(*ut)>::type T;
        if (!plan.nphase) return cudaSuccess;
        if (cudaMalloc(&ut, nch * (size_t)dof * sizeof(T)) != cudaSuccess ||
            cudaMalloc(&lam, nch * sizeof(T)) != cudaSuccess) {
            (void)cudaGetLastError();
            cudaFree(ut);
            ut = nullptr;
            plan.nphase = 0;
            return cudaSuccess;
        }
        slab_transpose_kernel<T><<<grid, 256>>>(F.d_U64, ut, g);
        const cudaError_t e = cudaGetLastError();
        return e != cudaSuccess ? e : cudaMemcpy(lam, host, nch * sizeof(T), cudaMemcpyHostToDevice);
    };
    CPMDP_CUDA(put(s->plan32, s->ut32, s->lam32, l32.data()));
    CPMDP_CUDA(put(s->plan64, s->ut64, s->lam64, F.lambda.data()));
    return CPMDP_OK;
}

cudaError_t malloc_any_time(void **p, size_t bytes) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaMalloc(p, bytes);
    cudaThreadExchangeStreamCaptureMode(&mode);
    return e;
}

void slab_workspace(const Factors &F, size_t elem) {
    if (!F.slab) return;
    DenseSlab &s = *F.slab;
    SlabPlan &plan = elem == 8 ? s.plan64 : s.plan32;
    void *&ws = elem == 8 ? s.ws64 : s.ws32;
    if (!plan.nphase || !plan.ws_bytes || ws) return;
    void *const other = elem == 8 ? s.ws32 : s.ws64;
    if (other && (elem == 8 ? s.plan32 : s.plan64).ws_bytes >= plan.ws_bytes) {
        ws = other;
    } else if (malloc_any_time(&ws, plan.ws_bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        ws = nullptr;
        plan.nphase = 0;
    }
}

const SlabPlan *slab_plan(const Factors &F, size_t elem) {
    if (!F.slab) return nullptr;
    const SlabPlan &p = elem == 8 ? F.slab->plan64 : F.slab->plan32;
    return p.nphase ? &p : nullptr;
}

template <typename T, int IB, int CB, int CBL>
static void slab_launch(const SlabArgs<T> &a, bool last, dim3 grid, cudaStream_t st) {
    const SlabPhase &p = a.p;
    if (p.nmodes <= 2) {
        if (last) slab_kernel<T, IB, CBL, true, 2><<<grid, p.threads, p.smem, st>>>(a);
        else slab_kernel<T, IB, CB, false, 2><<<grid, p.threads, p.smem, st>>>(a);
    } else {
        if (last) slab_kernel<T, IB, CBL, true, 0><<<grid, p.threads, p.smem, st>>>(a);
        else slab_kernel<T, IB, CB, false, 0><<<grid, p.threads, p.smem, st>>>(a);
    }
}

template <typename T>
cudaError_t slab_sweep(const Factors &F, const T *Vin, T *Vout, uint8_t *pi, int mode, T margin,
                       unsigned long long *res, unsigned *chg, const int *stop, cudaStream_t st) {
    constexpr bool f64 = sizeof(T) == 8;
    const DenseSlab &s = *F.slab;
    const SlabPlan &plan = f64 ? s.plan64 : s.plan32;
    const size_t S = (size_t)F.nstates;
    T *work = (T *)F.d_dense_work;
    SlabArgs<T> a;
    memset((void *)&a, 0, sizeof(a));
    a.ut = f64 ? (const T *)s.ut64 : (const T *)s.ut32;
    a.lam = f64 ? (const T *)s.lam64 : (const T *)s.lam32;
    a.ublock = plan.ublock;
    a.rank = F.rank;
    a.nact = F.nactions;
    a.mode = mode;
    a.gamma = (T)F.gamma;
    a.margin = margin;
    a.best = work;
    a.qold = work + S;
    a.arg = (uint8_t *)(work + 2 * S);
    a.R = f64 ? (const T *)F.d_R64 : (const T *)F.d_R32;
    a.Vin = Vin;
    a.Vout = Vout;
    a.pi = pi;
    a.res = res;
    a.changed = chg;
    a.stop = stop;
    for (int a0 = 0; a0 < F.nactions; a0 += plan.actions) {
        a.a0 = a0;
        a.a1 = std::min(F.nactions, a0 + plan.actions);
        a.c0 = a0 * F.rank;
        a.nchains = (a.a1 - a0) * F.rank;
        const size_t part = (size_t)plan.actions * F.rank * (size_t)plan.chain;
        a.ychain = plan.chain;
        const T *X = Vin;
        for (int i = 0; i < plan.nphase; i++) {
            const bool last = i == plan.nphase - 1;
            a.p = plan.ph[i];
            a.X = X;
            a.xchain = i == 0 ? 0 : plan.chain;
            a.ytiled = i == plan.nphase - 2;
            a.Y = last ? nullptr : (T *)(f64 ? s.ws64 : s.ws32) + (i & 1) * part;
            const SlabPhase &p = a.p;
            const long long nx = last ? (p.L + p.w - 1) / p.w : p.L * ((p.Rt + p.w - 1) / p.w);
            const dim3 grid((unsigned)nx, last ? 1u : (unsigned)((a.nchains + p.ch - 1) / p.ch));
            if (p.fine) slab_launch<T, f64 ? 1 : 2, f64 ? 2 : 4, f64 ? 2 : 4>(a, last, grid, st);
            else slab_launch<T, f64 ? 4 : 8, f64 ? 2 : 8, f64 ? 2 : 4>(a, last, grid, st);
            X = a.Y;
        }
    }
    return cudaGetLastError();
}

template cudaError_t slab_sweep<float>(const Factors &, const float *, float *, uint8_t *, int, float,
                                       unsigned long long *, unsigned *, const int *, cudaStream_t);
template cudaError_t slab_sweep<double>(const Factors &, const double *, double *, uint8_t *, int, double,
                                        unsigned long long *, unsigned *, const int *, cudaStream_t);

}  // namespace cpmdp
