// PM plan and driver shared by pm.cu and api.cu (internal).
#pragma once
#include <cufft.h>

#include "common.cuh"

namespace greem {
struct PmPlan {
    int n = 0;
    cufftHandle r2c = 0, c2r = 0;
    bool have = false;
};
int pm_plan(PmPlan &pl, int n, cudaStream_t s);
void pm_plan_destroy(PmPlan &pl);
// Complex values from one component's spectrum to the next (whole cache lines).
inline size_t pm_plane(int n) { return ((size_t)n * n * (n / 2 + 1) + 31) / 32 * 32; }
int run_pm(const PmPlan &pl, const double *pos, const float *mass, uint32_t N, double L, int n, int scheme, int pow2_e,
           const float *table, cufftComplex *tmp, float4 *field, float *acc, int accumulate, cudaStream_t s, int nsm);
}  // namespace greem
