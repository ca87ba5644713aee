// H psi for a Pauli sum H (kernels_hpsi.cu): the adjoint's costate seed, the
// exact solvers' derivative.
#pragma once

#include <memory>

#include "internal.h"

namespace qsim {

// A (possibly strided) batch of n-qubit states: member b starts at amplitude b << ms.
struct StateView {
    void *data;
    int n;
    int ms;
    int batch;
    qs_dtype dtype;
};

// A Pauli sum prepared for states of one shape (grouped by X mask, coefficients
// in the state's precision, one parameter block per launch); it may be applied
// any number of times, to any states of that shape.
struct HpsiOp {
    struct Impl;
    std::shared_ptr<Impl> impl;
};
qs_status hpsi_prepare(const StateView &shape, const qs_pauli_term *terms, size_t count, HpsiOp *op);

// One result of an application: out = base + c (H src), or c (H src) where base
// is null. out may be base; neither out may be src.
struct HpsiOut {
    void *out = nullptr;  // null: no such result
    const void *base = nullptr;
    cd c = 1.0;
};
// Up to two results of one application. A sum that takes several launches (very
// many terms) keeps its partial sums in `spare`, one state of src's shape and
// stride that is neither src nor a base; it may be an output.
qs_status hpsi_apply(const HpsiOp &op, const StateView &src, const HpsiOut &a, const HpsiOut &b, void *spare,
                     cudaStream_t st);

// dst = H src
qs_status k_pauli_apply(const StateView &src, const StateView &dst, const qs_pauli_term *terms, size_t count,
                        cudaStream_t st);

}  // namespace qsim
