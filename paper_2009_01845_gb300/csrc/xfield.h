// Expectation of a transverse field (kernels_xfield.cu).
#pragma once

#include "internal.h"

namespace qsim {

// Whether the fused kernel takes the `terms` single-X terms of a state of n
// qubits: the state spans one of its tiles, and there are at least two (one
// term is one read of the state either way; at n = 27 complex64, 0.18 ms).
bool xfield_fits(int n, int terms);

// sum_b coeff[b] <X on index bit b> per member, as `blocks` partial sums
// part[member * blocks + i] (double2: the sum and 0), added to what part holds
// if `accumulate`. coeff: one entry per index bit, 0 for none, at least one
// nonzero.
qs_status k_xfield(const void *psi, int n, int ms, int batch, qs_dtype dtype, const double *coeff, void *part,
                   int blocks, bool accumulate, cudaStream_t st);

}  // namespace qsim
