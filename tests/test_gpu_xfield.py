"""GPU parity of the energy of a transverse field, whose X terms run several
per read of the state: tile edges (n = 11: below a tile, 12: one tile, 13: one
window bit that overlaps the tile, 20, 21, 22: a full window and one bit more),
uneven and missing coefficients, X terms beside Z strings on the same qubit,
batches, and the allocation-free entry point.

Tolerance: the sums of 16 products in the state's precision u lose at most
16 u sum|c| of a normalised state, twice over (products and coefficients)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu

UNIT = {"c128": 2.0 ** -53, "c64": 2.0 ** -24}


def field(n, seed):
    r = qi.rng(seed)
    terms = [(float(r.normal()), 1 << q, 0) for q in range(n) if q % 5 != 3]
    terms += [(float(r.normal()), 1 << 0, 0)]                    # a second X on qubit 0
    terms += [(0.4, 1 << (n - 1), 1 << 1), (-0.3, 1 << 2, 1 << 2)]  # X Z and Y: not plain X groups
    terms += [(float(r.normal()), 0, (1 << i) | (1 << (i + 1))) for i in range(n - 1)]
    return terms


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,batch", [(11, 2), (12, 3), (13, 1), (20, 2), (21, 1), (22, 1)])
def test_field_energy_matches_oracle(dtype, n, batch):
    import torch
    from paper_2009_01845_gb300 import qsim
    lib = qsim.load(build_if_missing=True)
    psis = np.stack([qi.random_state(n, 500 + 10 * n + b) for b in range(batch)])
    st = qsim.State(n, batch=batch, dtype=dtype).set(psis)
    held = st.get().reshape(batch, -1).astype(np.complex128)
    terms = field(n, n)
    tol = 64 * UNIT[dtype] * sum(abs(t[0]) for t in terms)
    got = st.expectation(terms)
    out = torch.full((2 * batch,), float("nan"), dtype=torch.float64, device="cuda")
    arr, cnt = qsim.marshal_terms(terms)
    assert lib.qs_expectation_noalloc(ctypes.c_void_p(st.tensor.data_ptr()), n, batch, qsim.DTYPE[dtype], arr, cnt,
                                      ctypes.c_void_p(out.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    o = out.cpu().numpy().reshape(batch, 2)
    for b in range(batch):
        want = oracle.expectation(np.ascontiguousarray(held[b]), n, terms)
        assert abs(got[b] - want) <= tol
        assert abs(o[b, 0] + 1j * o[b, 1] - want) <= tol
