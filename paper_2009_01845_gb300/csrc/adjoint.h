// Adjoint gradient: shared declarations of its kernels and driver.
#pragma once

#include "device.cuh"
#include "hpsi.h"
#include "internal.h"

namespace qsim {

constexpr int kGRMaxRows = 1024;   // parameters per reduction launch
constexpr int kGRMaxSlots = 2048;  // gradient slots per reduction launch

struct GradReduceP {
    int beg[kGRMaxRows + 1];   // slot list of parameter row i: slot[beg[i] .. beg[i+1])
    int slot[kGRMaxSlots];
    float coef[kGRMaxSlots];   // 1 for rotations (Im<l|P|phi>), -2 for phase gates
    uint64_t total_tiles;
    uint64_t tiles_per_member;
    int n_params;
    int param0;                // first parameter row of this launch
};

qs_status k_dot(const StateView &a, const StateView &b, double *scratch, size_t scratch_doubles, double *out,
                cudaStream_t st);
qs_status k_grad_reduce(const double *part, const GradReduceP &p, int n_param_rows, int batch, double *grad,
                        cudaStream_t st);

}  // namespace qsim
