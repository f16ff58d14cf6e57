// Host check of which dense models get a plan of fused sweeps (dense_slab.cu over the
// allocator of fake_cudart.cpp, no GPU). Prints one line per check that fails; exit code 1
// when there are any.
#include "dense_slab.cu"

#include <stdio.h>

namespace cpmdp {
void set_error(const char *, ...) {}
cpmdp_status cuda_fail(cudaError_t, const char *) { return CPMDP_ECUDA; }
}  // namespace cpmdp

using namespace cpmdp;

int main() {
    // actions, rank, shape; a plan in FP32, in FP64
    const int models[][7] = {{1, 1, 1500, 0, 0, 0, 1}, {2, 1, 1500, 0, 0, 0, 1}, {2, 1, 2, 1500, 0, 0, 1}, {2, 1, 2000, 0, 0, 0, 0},
                             {2, 1, 2500, 4, 0, 0, 0}, {4, 3, 1500, 0, 0, 1, 1}, {2, 1, 1500, 32, 0, 1, 1}, {2, 1, 1000, 0, 0, 1, 1},
                             {4, 3, 1000, 500, 0, 1, 1}, {8, 8, 64, 64, 64, 1, 1}, {4, 3, 8, 8, 8, 1, 1}};
    int failed = 0;
    for (const auto &m : models) {
        Factors F;
        F.num_sms = 152;
        F.nactions = m[0];
        F.rank = m[1];
        F.nstates = 1;
        for (F.ndim = 0; F.ndim < 3 && m[2 + F.ndim]; F.ndim++) {
            F.shape[F.ndim] = m[2 + F.ndim];
            F.nstates *= m[2 + F.ndim];
        }
        F.lambda.assign((size_t)F.nactions * F.rank, 1.0);
        if (slab_prepare(F) != CPMDP_OK) failed = 1;
        for (int k = 0; k < 2; k++)
            if ((slab_plan(F, k ? 8 : 4) != nullptr) != (m[5 + k] != 0)) {
                failed = 1;
                printf("A %d R %d, %d x %d x %d, %s: plan %d expected\n", m[0], m[1], m[2], m[3], m[4], k ? "FP64" : "FP32", m[5 + k]);
            }
        slab_free(F);
    }
    return failed;
}
