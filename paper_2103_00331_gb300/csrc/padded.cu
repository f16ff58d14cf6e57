// FP32 GridWorld solves of grids whose rows are not a multiple of 4 states.
//
// The solvers' 16-byte loads, and the barrier-free solver as a whole, need
// rows of whole 4-state segments; other rows ran one state a thread with a
// grid barrier per sweep. Such a grid is solved on a copy with its rows padded
// by obstacle states (value 0, never entered: the moves off the row's end are
// walls in the codes already, and obstacles take no part in the residual), so
// every real state sees the same neighbours and the same arithmetic: values,
// policies, sweep counts and residuals are those of the unpadded solve. Two
// small kernels copy the values in and the results out.
#include <algorithm>
#include <new>

#include "banded_common.cuh"
#include "flow.h"
#include "march.h"

namespace cpmdp {

struct PadGeom {
    int n, pitch;              // row length and its padded length
    int total;                 // padded states
};

// out[row pitch + c] = in[row n + c], pads = fill; elements of T.
template <typename T>
__global__ void pad_rows_kernel(const T *__restrict__ in, T *__restrict__ out, PadGeom g, T fill) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.total; i += gridDim.x * blockDim.x) {
        const unsigned row = (unsigned)i / (unsigned)g.pitch;
        const int c = i - (int)(row * (unsigned)g.pitch);
        out[i] = c < g.n ? in[(size_t)row * g.n + c] : fill;
    }
}

// Values and policy of the real states (either may be null).
__global__ void unpad_kernel(const float *__restrict__ Vp, const uint8_t *__restrict__ pip, float *__restrict__ V,
                             uint8_t *__restrict__ pi, PadGeom g) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.total; i += gridDim.x * blockDim.x) {
        const unsigned row = (unsigned)i / (unsigned)g.pitch;
        const int c = i - (int)(row * (unsigned)g.pitch);
        if (c >= g.n) continue;
        const size_t s = (size_t)row * g.n + c;
        if (V) V[s] = Vp[i];
        if (pi) pi[s] = pip[i];
    }
}

static int grid_of(const Factors &F, int n) { return std::max(1, std::min((n + 255) / 256, F.num_sms * 8)); }

static PadGeom geom_of(const Factors &F) {
    const int n = (int)F.shape[F.ndim - 1];
    return {n, (n + 3) & ~3, (int)(F.nstates / n * ((n + 3) & ~3))};
}

// Padded copies of at least kMarchMinStates and less than this run their value
// iteration and their certificate without the marching sweep (pad_grid_barrier).
constexpr int64_t kPadMarchStates = 28ll << 20;

bool pad_wanted(const Factors &F, cpmdp_precision prec, bool policy_iteration, const SolveOpts &o) {
    if (F.kind != CPMDP_GRIDWORLD || prec != CPMDP_F32 || o.fused != 1 || o.inject_stall) return false;
    const int64_t n = F.shape[F.ndim - 1], pitch = (n + 3) & ~3ll;
    // Up to 256 states one block solves the grid (30 us of 38 sweeps in all).
    // The copies cost about 8 us a solve, the pads their share of every sweep,
    // so rows grow by a third at most; with four dimensions and more, where
    // only the vector loads are won, 9 x 8 x 7 x 5 x 6 took 173 us padded, 140 as
    // it is. Measured: value iteration at 300 x 301 461 -> 250 us, at
    // 67 x 65 x 66 722 -> 406 us, at 101 x 97 x 103 (past the barrier-free
    // solver's size) 1,230 -> 925 us; policy iteration there 1,443 -> 1,407 us.
    if (n % 4 == 0 || F.ndim > 3 || F.nstates <= 256 || F.nstates / n * pitch >= (1ll << 30)) return false;
    if (pitch * 3 > n * 4) return false;
    // A solve limited to a few sweeps ends before they have paid for the copies:
    // one sweep at 301 x 299 45 us as it is, 61 padded; 12 sweeps 69 and 69, 24
    // sweeps 92 and 80; 55 x 56 x 57 78 and 84 at 12 sweeps, 91 and 90 at 16. From
    // 101 x 97 x 103 on one sweep pays (93 and 88).
    const int64_t eval = std::min(o.partial_eval, o.max_eval_iter);
    const int64_t sweeps = !policy_iteration ? o.max_iter : o.partial_eval > 0 ? o.max_rounds * (eval + 1) : 1ll << 40;
    return sweeps >= 12 || F.nstates >= 800000;
}

// Columns of four segments make the barrier-free policy iteration of
// three-dimensional grids slower than the grid barrier (20 rounds at 75 x 73 x
// 74: 349 and 301 us, 326 on the rows as they are; two dimensions 248 and 292 at
// 751 x 749). Up to 28 million states the grid barrier's 16-byte sweeps are
// faster than the marching sweep: 100 sweeps at 203 x 207 x 209 3,694 and 4,597
// us (4,004 on the rows as they are), 259 x 255 x 257 6,778 and 8,374 (7,512),
// 321 x 319 x 318 11,810 and 10,812 (13,805).
bool pad_grid_barrier(const Factors &P, bool policy_iteration) {
    if (P.ndim != 3) return false;
    return policy_iteration ? flow_column(P, true) == 4 : P.nstates >= kMarchMinStates && P.nstates < kPadMarchStates;
}

// The same sizes take the FP64 certificate on the rows as they are: 224 us less
// at 203 x 207 x 209, 368 at 259 x 255 x 257, 93 at 321 x 319 x 318; 94 more at
// 361 x 359 x 357, and 104 more at 189 x 190 x 191, which does not march.
bool pad_certify_rows(const Factors &P) {
    return P.ndim == 3 && P.nstates >= kMarchMinStates && P.nstates < kPadMarchStates;
}

void pad_free(Factors &F) {
    if (!F.pad) return;
    if (F.pad->march_graph) cudaGraphExecDestroy(F.pad->march_graph);
    if (F.pad->d_arena) cudaFreeAsync(F.pad->d_arena, 0);
    delete F.pad;
    F.pad = nullptr;
}

cpmdp_status pad_prepare(Factors &F, cudaMemPool_t pool, cudaStream_t st) {
    if (F.pad) return CPMDP_OK;
    Factors *P = new (std::nothrow) Factors;
    if (!P) { set_error("out of host memory"); return CPMDP_ENOMEM; }
    const PadGeom g = geom_of(F);
    P->device = F.device;
    P->kind = F.kind;
    P->ndim = F.ndim;
    for (int d = 0; d < F.ndim; d++) P->shape[d] = F.shape[d];
    P->shape[F.ndim - 1] = g.pitch;
    int64_t stride = 1;
    for (int d = F.ndim - 1; d >= 0; d--) {
        P->stride[d] = stride;
        stride *= P->shape[d];
    }
    P->nstates = stride;
    P->nactions = F.nactions;
    P->rank = F.rank;
    P->p = F.p;
    P->gamma = F.gamma;
    P->w_move = F.w_move;
    P->w_perp = F.w_perp;
    P->w_stay = F.w_stay;
    P->code_bytes = F.code_bytes;
    P->num_sms = F.num_sms;
    P->d_ctrl = F.d_ctrl;
    const size_t S = (size_t)P->nstates;
    auto up = [](size_t n) { return (n + 255) & ~(size_t)255; };
    const bool flow = flow_shape_ok(*P);
    const size_t o_R32 = up(S * sizeof(double)), o_W = o_R32 + up(S * sizeof(float)), o_V = o_W + up(S * sizeof(float));
    const size_t o_code = o_V + up(S * sizeof(float)), o_pi = o_code + up(S), o_flow = o_pi + up(S);
    const size_t total = o_flow + (flow ? up(flow_bytes(*P)) : 0);
    cudaError_t e = cudaMallocFromPoolAsync(&P->d_arena, total, pool, st);
    if (e != cudaSuccess) {
        delete P;
        (void)cudaGetLastError();
        set_error("no device memory for the padded rows");
        return CPMDP_ENOMEM;
    }
    char *arena = static_cast<char *>(P->d_arena);
    P->d_R64 = reinterpret_cast<double *>(arena);
    P->d_R32 = reinterpret_cast<float *>(arena + o_R32);
    P->d_scratch = arena + o_W;
    P->scratch_bytes = S * sizeof(float);
    P->pad_V = reinterpret_cast<float *>(arena + o_V);
    P->d_code = arena + o_code;
    P->pad_pi = reinterpret_cast<uint8_t *>(arena + o_pi);
    const int grid = grid_of(F, g.total);
    const uint8_t wall = (uint8_t)((1u << (2 * F.ndim)) - 1 | 1u << (2 * F.ndim));   // an obstacle's code
    pad_rows_kernel<double><<<grid, 256, 0, st>>>(F.d_R64, P->d_R64, g, 0.0);
    pad_rows_kernel<float><<<grid, 256, 0, st>>>(F.d_R32, P->d_R32, g, 0.f);
    // codes of at most three dimensions (pad_wanted) are one byte
    pad_rows_kernel<uint8_t><<<grid, 256, 0, st>>>((const uint8_t *)F.d_code, (uint8_t *)P->d_code, g, wall);
    e = cudaGetLastError();
    if (e == cudaSuccess && flow) {
        P->d_flow = arena + o_flow;
        P->flow_in_arena = true;
        e = cudaMemsetAsync(static_cast<char *>(P->d_flow) + flow_counter_bytes(), 0xFF,
                            flow_bytes(*P) - flow_counter_bytes(), st);
    }
    if (e != cudaSuccess) {
        cudaFreeAsync(P->d_arena, st);
        delete P;
        return cuda_fail(e, "padded rows");
    }
    F.pad = P;
    return CPMDP_OK;
}

cudaError_t pad_in(const Factors &F, const float *V, cudaStream_t st) {
    const PadGeom g = geom_of(F);
    pad_rows_kernel<float><<<grid_of(F, g.total), 256, 0, st>>>(V, F.pad->pad_V, g, 0.f);
    return cudaGetLastError();
}

cudaError_t pad_out(const Factors &F, float *V, uint8_t *pi, cudaStream_t st) {
    const PadGeom g = geom_of(F);
    unpad_kernel<<<grid_of(F, g.total), 256, 0, st>>>(F.pad->pad_V, F.pad->pad_pi, V, pi, g);
    return cudaGetLastError();
}

}  // namespace cpmdp
