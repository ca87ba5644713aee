// Gate queues on states below a tile (kernels_small.cu).
#pragma once

#include <vector>

#include "internal.h"

namespace qsim {

// Whether a state of n qubits is one the small-state kernel holds (the widths
// the tiled passes do not take).
bool small_state(const qs_state *s);
// Whether the kernel takes the queue in place of a launch per gate: the state is
// one it holds, and gates and members are ones it is the faster form for.
bool one_launch(const qs_state *s, const std::vector<LGate> &G);

// Apply the queue to every member, in as few launches as its descriptors need.
// Batched-parameter gates take angle * param_sign; gradient ops (kind
// kKindGrad, the adjoint sweep: the top index bit tells phi from lambda) write
// gpart[slot * batch + member].
qs_status run_small(qs_state *s, const std::vector<LGate> &G, const double *params, int n_params,
                    double param_sign = 1.0, double *gpart = nullptr);

}  // namespace qsim
