"""What a marginal's sums hold (complex64): the products added in FP32 before an
FP64 sum are those of amplitudes that differ in the bits between 8 and the
group's lowest bit above them (none where that is bit 8). Here at most one of
them is nonzero, and all values are dyadic with exact FP64 sums, so the
probabilities are equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lowest", [8, 9, 10, 11])
@pytest.mark.parametrize("others", [(), (0, 3), (6, 7, 13), (14, 15)])
def test_short_runs_are_summed_in_fp64(lowest, others):
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    n = 16
    x = np.arange(1 << n)
    psi = np.where((x >> 8) % 32 == 0, 1.0, 2.0 ** -13)
    psi[(x >> 8) & ((1 << (lowest - 8)) - 1) != 0] = 0.0
    bits = sorted((lowest,) + others, reverse=True)  # the group's qubits, the outcome's bits from the top
    y = sum(((x >> b) & 1) << (len(bits) - 1 - j) for j, b in enumerate(bits))
    want = np.bincount(y, weights=psi * psi, minlength=1 << len(bits))
    got = qsim.State(n).set(psi).marginal_probabilities([n - 1 - b for b in bits])
    np.testing.assert_array_equal(got, want)
