// Host side of the banded factorisation of large blocks (band.cu): Cholesky, W = L^-1 [J^T b]
// and, in FP64, the map D = W^T W, c = W^T g, each as one launch over all such blocks of a grid
// scene.  Internal to libsubadmm.
#pragma once

#include <cuda_runtime.h>

#include <vector>

namespace subadmm {

constexpr int kBandMax = 384;          // widest envelope (largest p - env[p]) taken
constexpr int kBandThreads = 256;
constexpr int kBandCols = 32;          // columns of W per block

// One block's K_i (FP32 or FP64, by the launch)
struct BandJob {
    void *K;                  // n x n row-major, lower triangle inside the envelope: K, then its
                              // factor.  FP32: 1 / L_pp ends on the diagonal; FP64: L_pp
    void *LT;                 // FP64: copy of the factor with 1 / L_pp on the diagonal
    double *idg;              // FP64: 1 / L_pp
    const int *env, *lastr;   // first column of row p inside the envelope; last row that column
                              // k reaches (both nondecreasing)
    const int *jlo, *jhi;     // columns [jlo, jhi) of row t of J
    const double *J, *b;      // J m x n, b n
    void *W;                  // n rows of ldw: column t < m is L^-1 J^T e_t, column m is L^-1 b
    void *D, *c;              // FP64: D rows ldd apart (zero from m to mpad), c
    int n, m, ldw, ldd, mpad;
    int *pending;             // step flag: taken while it is 4; cleared on failure
    int *subflag;             // kept-factor flag, cleared on failure (null: none)
};

struct BandPlan {
    int device = -1;
    bool fp64 = false;
    int njobs = 0, nw = 0, nd = 0;     // jobs, tasks of W, tasks of D
    int bw = 0;                        // widest envelope of the jobs
    int cluster = 1;                   // blocks per matrix in the factorisation
    BandJob *d_jobs = nullptr;
    int2 *d_w = nullptr;               // job, first column
    int4 *d_d = nullptr;               // job, row tile, column tile, first row of W that matters
    int *status = nullptr;             // set on a non-positive pivot
    int fail_status = 0;
};

// jobs with device pointers; jlo: each job's jlo on the host (its tasks' order and extents)
cudaError_t band_plan_build(BandPlan &P, const std::vector<BandJob> &jobs,
                            const std::vector<std::vector<int>> &jlo, int bw, bool fp64, int *status,
                            int fail_status);
cudaError_t band_plan_run(const BandPlan &P, cudaStream_t st);
void band_plan_free(BandPlan &P);

}  // namespace subadmm
