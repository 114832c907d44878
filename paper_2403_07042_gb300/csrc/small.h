// FP64 steps of small models, many in one launch of one thread-block cluster (small.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "model.h"

namespace qed {

// Three D x D matrices fit an SM's shared memory up to 64 states.
constexpr int kSmallMaxDim = 64;
constexpr int kSmallMaxCtas = 16;
constexpr int kSmallStepsPerLaunch = 4096;

struct SmallModel {
    int D = 0, ctas = 1, rows = 1;  // rows of the result a CTA takes
    size_t smem = 0;
    void *block = nullptr;  // the allocation of the tables below
    int *ptr = nullptr, *idx = nullptr;  // states of row i's component: idx[ptr[i] .. ptr[i + 1])
    // of the model, filled in at launch
    const double2 *U = nullptr;
    double dt = 0.0;
    const double *anti = nullptr, *in_coef = nullptr;
    const int32_t *in_ptr = nullptr, *in_jump = nullptr, *in_src = nullptr;
};

// Sets m->small (null before) where a cluster run pays (and the device can hold the cluster), with the
// components of H's graph, or every state for every row (`whole`: an injected U).
qed_status small_prepare(qed_model *m, bool whole, const std::vector<int> &component);
void small_release(SmallModel *a);
// What a run records: the observables ids[0 .. n_obs) (as qed_evolve's) at every step whose
// number, counted from `first`, is a multiple of `every`; rows of `out` from `row` on.
struct SmallRecords {
    int n_obs = 0, every = 1, from_start = 0;
    int64_t row = 0;
    const int32_t *ids = nullptr;
    const double *weights = nullptr;
    double *out = nullptr;
};

// qed_evolve's steps and records of rho (device, D x D, in place), Lie or effective; the ids
// are in m->obs_ids_dev.
qed_status small_run(qed_model *m, double2 *rho, int64_t steps, int64_t offset, int32_t every, int32_t n_obs,
                     double *out, cudaStream_t s);

}  // namespace qed
