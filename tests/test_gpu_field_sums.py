"""What the sums of a transverse field's energy hold (complex64): every term of
a thread as FP64 would, products one by one in FP64 where a state is one tile
(n = 12), infinities and sums beyond the range of floats as FP64 gives them. All
values are dyadic and their FP64 sums exact in any order, so results are equal."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def energies(n, psi, terms):
    import torch
    from paper_2009_01845_gb300 import qsim
    lib = qsim.load(build_if_missing=True)
    st = qsim.State(n).set(psi)
    out = torch.full((2,), float("nan"), dtype=torch.float64, device="cuda")
    arr, cnt = qsim.marshal_terms(terms)
    assert lib.qs_expectation_noalloc(ctypes.c_void_p(st.tensor.data_ptr()), n, 1, qsim.DTYPE["c64"], arr, cnt,
                                      ctypes.c_void_p(out.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return [float(st.expectation(terms)[0].real), float(out[0])]


def x_on(n, coeff, bit):
    return (coeff, 1 << (n - 1 - bit), 0)


@pytest.mark.parametrize("n", [13, 16])
def test_small_terms_are_kept_beside_large_ones(n):
    c = [1.0, 2.0 ** -24, 2.0 ** -48]
    for bits in ((8, 4, 0), (0, 4, 8), (3, 2, 1)):
        got = energies(n, np.ones(1 << n), [x_on(n, v, b) for v, b in zip(c, bits)])
        assert got == [2.0 ** n * sum(c)] * 2


def test_products_of_one_tile_are_summed_in_fp64():
    n = 12
    psi = np.full(1 << n, 2.0 ** -13)
    psi[0] = psi[1 << 9] = 1.0
    x = np.arange(1 << n)
    want = float(sum(c * np.sum(psi * psi[x ^ (1 << b)]) for c, b in ((1.0, 9), (0.5, 5), (0.25, 1))))
    assert energies(n, psi, [x_on(n, 1.0, 9), x_on(n, 0.5, 5), x_on(n, 0.25, 1)]) == [want] * 2


def test_sums_beyond_floats():
    n = 13
    terms = [x_on(n, 1.0, b) for b in range(n)]
    assert energies(n, np.full(1 << n, 2.0 ** 61), terms) == [n * 2.0 ** (n + 122)] * 2
    assert energies(n, np.full(1 << n, 1e20), terms) == [np.inf] * 2
