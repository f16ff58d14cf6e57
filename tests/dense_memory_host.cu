// Host check of what dense models ask of the CUDA runtime: dense_slab.cu over the
// allocator of fake_cudart.cpp (no GPU). Prints one line per check that fails; exit code 1
// when there are any.
#include "dense_slab.cu"

#include <stdio.h>

namespace cpmdp {
void set_error(const char *, ...) {}
cpmdp_status cuda_fail(cudaError_t, const char *) { return CPMDP_ECUDA; }
}  // namespace cpmdp

extern size_t held;        // fake_cudart.cpp
extern int allow;
extern bool capturing, relaxed;

using namespace cpmdp;

static int failed = 0;
static void check(bool ok, const char *what, const Factors &F) {
    if (ok) return;
    failed = 1;
    printf("%s: A %d R %d, %lld states\n", what, F.nactions, F.rank, (long long)F.nstates);
}

int main() {
    const int models[][6] = {{8, 8, 64, 64, 64, 64}, {4, 4, 48, 50, 52, 46}, {64, 64, 41, 41, 41, 0}, {6, 49, 85, 99, 104, 0},
                             {6, 4, 52, 50, 54, 56}, {20, 8, 118, 118, 133, 0}, {4, 3, 8, 8, 8, 8}, {2, 2, 5, 0, 0, 0}};
    for (const auto &m : models) {
        Factors F;
        F.num_sms = 152;
        F.nactions = m[0];
        F.rank = m[1];
        F.nstates = 1;
        size_t padded = 0;
        for (F.ndim = 0; F.ndim < 4 && m[2 + F.ndim]; F.ndim++) {
            const int64_t n = m[2 + F.ndim];
            F.shape[F.ndim] = n;
            F.nstates *= n;
            padded += (size_t)((n + 3) & ~3) * ((n + 7) & ~7);
        }
        const size_t chains = (size_t)F.nactions * F.rank, factors = chains * (padded + 1) * 12;
        F.lambda.assign(chains, 1.0);
        // the build takes the transposed factors and nothing else
        check(slab_prepare(F) == CPMDP_OK, "build", F);
        check(held == factors, "the build holds more than its factors", F);
        for (size_t elem : {4, 8}) {
            const SlabPlan *p = slab_plan(F, elem);
            check(p != nullptr, "a plan", F);
            // 1 GiB a buffer, or one action
            const size_t action = (size_t)F.rank * (size_t)p->chain * elem, bufs = p->nphase > 2 ? 2 : 1;
            check(p->ws_bytes <= bufs * std::max<size_t>(1u << 30, action), "intermediates past their bound", F);
            check(p->nphase < 2 || p->ws_bytes == bufs * action * p->actions, "workspace of the group", F);
        }
        // each precision takes its own share, also under a capture; an earlier one that is large enough serves both
        capturing = true;
        slab_workspace(F, 4);
        check(held == factors + slab_plan(F, 4)->ws_bytes, "workspace of FP32 sweeps", F);
        slab_workspace(F, 4);
        slab_workspace(F, 8);
        capturing = false;
        check(!relaxed, "the thread's capture mode", F);
        const size_t w4 = slab_plan(F, 4)->ws_bytes, w8 = slab_plan(F, 8)->ws_bytes;
        check(held == factors + w4 + (w4 >= w8 ? 0 : w8), "workspace of both", F);
        check(!w4 || F.slab->ws32, "FP32 workspace", F);
        check(!w8 || F.slab->ws64, "FP64 workspace", F);
        slab_free(F);
        check(held == 0, "memory given back", F);
        // without the memory for its workspace a sweep has no plan
        check(slab_prepare(F) == CPMDP_OK, "build", F);
        allow = 0;
        slab_workspace(F, 8);
        slab_workspace(F, 4);
        allow = -1;
        check(!w8 || !slab_plan(F, 8), "FP64 plan dropped", F);
        check(!w4 || !slab_plan(F, 4), "FP32 plan dropped", F);
        slab_free(F);
        check(held == 0, "memory given back after a failure", F);
        // nor does the build fail without the memory for its factors, whichever of them is refused
        for (int n = 0; n < 4; n++) {
            allow = n;
            check(slab_prepare(F) == CPMDP_OK, "build without memory", F);
            allow = -1;
            check((slab_plan(F, 4) != nullptr) == (n >= 2), "FP32 plan without its factors", F);
            check(!slab_plan(F, 8), "FP64 plan without its factors", F);
            slab_free(F);
            check(held == 0, "memory given back after a failed build", F);
        }
    }
    return failed;
}
