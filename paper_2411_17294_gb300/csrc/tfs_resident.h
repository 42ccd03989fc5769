// Many steps of the pointwise law in one launch (FP32 storage, the stress form,
// alpha < 1, BDF2 start, frozen velocity gradient): tfs_resident.cu.
#pragma once

#include "tfs_internal.h"

namespace tfs {

constexpr int kRunSteps = 128;   // steps one launch takes (their scalars travel as kernel parameters)

struct ResidentRun {
    const float* kap;      // [d*d][N]
    const float* sigma0;   // [nc][N] or nullptr
    float* modes_n;        // levels n and n-1, tile-major (mode_index), advanced in place
    float* modes_nm1;
    float* rows;           // sigma^{n+1} of step k at rows + k stride (elements)
    long long stride;
    unsigned* flags;
    long long N;
    int m, steps;
    ModeConstsF mc;
    F2c eta, a, dt;
    F2c src[kRunSteps];    // dt G g_alpha
};
cudaError_t launch_resident_run(const ResidentRun& a, int dim, bool compensated, cudaStream_t s);

struct ResidentBack {
    const float* kap;
    const float* rows;     // sigma^{n+1} of the steps, in time order as above
    long long stride;
    const float* dJ;       // adjoint of the stress after the last of these steps (nullptr: none but its modes')
    float* ell_prev;       // adjoint mode levels of the two later steps, tile-major, advanced in place
    float* ell_prev2;
    double* g_sigma0;      // added to
    double* g_kap;
    double* partials;      // [2 tile], [2 tile + 1] added to
    unsigned* flags;
    long long N;
    int m, steps;
    ModeConstsF mc;
    float a, dt;
    double eta, dt_wi2, g_wi, inv_wire;   // eta, dt/Wi^2, G/Wi, 1/(Wi Re)
    float src[kRunSteps];            // dt G g_alpha
    double dtg[kRunSteps];           // dt g_alpha
};
cudaError_t launch_resident_back(const ResidentBack& a, int dim, cudaStream_t s);

}  // namespace tfs
