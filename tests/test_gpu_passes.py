"""GPU parity of tiled passes on what specialised kernels treat apart: 2-qubit
gates and SWAPs on the low index bits (in the tile, any stage), diagonal blocks
of signs alone, of uniform phases and of phases that vary between threads, and
long runs of stages over one and several tiles (transposes inside warps and
across them, tile after tile). Generic and specialised kernels, both
precisions, against the oracle at the scope's bounds; SWAPs of complex128
amplitudes alone are exact."""
import numpy as np
import pytest

import oracle
from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu

TOL = {"c128": (1e-12, 1e-11), "c64": (1e-5, 1e-4)}


@pytest.fixture(scope="module")
def qs():
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    yield qsim
    qsim.jit_set_policy("tiered")


def low_two_qubit(n, r):
    g = []
    for k in range(40):
        a, b = (int(x) for x in r.permutation(6)[:2])          # index bits 0 .. 5
        q = (n - 1 - a, n - 1 - b)
        g.append(qi.Gate("SWAP", q) if k % 3 == 0 else qi.Gate("UNITARY", q, (), (), qi.random_unitary(2, r)))
        far = int(r.integers(0, n - 6))
        g.append(qi.Gate("UNITARY", (far, n - 1 - int(r.integers(0, 5))), (), (), qi.random_unitary(2, r)))
        g.append(qi.Gate("U3", (int(r.integers(0, n)),), (), tuple(float(v) for v in r.uniform(0, 6.28, 3))))
    return g


def diagonals(n, r):
    g = []
    for layer in range(8):
        for q in range(n):
            if layer % 2:
                g.append(qi.Gate("RY", (q,), (), (float(r.uniform(0, 6.28)),)))
            else:
                g.append(qi.Gate("U3", (q,), (), tuple(float(v) for v in r.uniform(0, 6.28, 3))))
        for q in range(n - 1):
            g.append(qi.Gate("CZ", (q, q + 1)))
        for q in range(layer % 3, n - 2, 3):
            g.append(qi.Gate("CZ", (q, q + 2), ((q + 1),)))
            if layer % 4 == 1:
                g.append(qi.Gate("CU1", (q, q + 2), (), (float(r.uniform(0, 6.28)),)))
    return g


@pytest.mark.parametrize("policy", ["off", "sync"])
@pytest.mark.parametrize("dtype,n", [("c64", 13), ("c64", 15), ("c128", 12), ("c128", 15)])
@pytest.mark.parametrize("circuit", [low_two_qubit, diagonals])
def test_pass_kernels(qs, circuit, dtype, n, policy):
    gates = circuit(n, qi.rng(17 * n))
    psi = qi.random_state(n, n)
    want = oracle.apply_circuit(psi.copy(), n, gates)
    qs.jit_set_policy(policy)
    got = qs.State(n, dtype=dtype).set(psi).apply(gates, mode="tiled").get()
    mx, l2 = TOL[dtype]
    assert np.max(np.abs(got - want)) <= mx and np.linalg.norm(got - want) <= l2


@pytest.mark.parametrize("n", [5, 12, 14])
def test_low_swaps_of_complex128_are_exact(qs, n):
    gates = [qi.Gate("SWAP", (n - 1, n - 4)), qi.Gate("SWAP", (n - 2, n - 1))]
    psi = qi.random_state(n, 3) * 2.0 ** qi.rng(1).integers(-300, 1, size=1 << n)
    want = oracle.apply_circuit(psi.copy(), n, gates)
    got = qs.State(n, dtype="c128").set(psi).apply(gates).get()
    np.testing.assert_array_equal(got, want)
