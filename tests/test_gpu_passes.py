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


# complex128 circuits are short: a specialised double-float pass takes seconds
# to compile, one with 4x4 gates far longer
def low_two_qubit(n, r, long):
    g = []
    for k in range(12 if long else 3):
        a, b = (int(x) for x in r.permutation(6)[:2])          # index bits 0 .. 5
        q = (n - 1 - a, n - 1 - b)
        g.append(qi.Gate("SWAP", q) if k % 3 == 0 else qi.Gate("UNITARY", q, (), (), qi.random_unitary(2, r)))
        far = int(r.integers(0, n - 6))
        g.append(qi.Gate("UNITARY", (far, n - 1 - int(r.integers(0, 5))), (), (), qi.random_unitary(2, r)))
        g.append(qi.Gate("U3", (int(r.integers(0, n)),), (), tuple(float(v) for v in r.uniform(0, 6.28, 3))))
    return g


def diagonals(n, r, long):
    g = []
    for layer in range(8 if long else 2):
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
@pytest.mark.parametrize("dtype,n,fp64", [("c64", 13, False), ("c64", 15, False), ("c128", 12, False),
                                          ("c128", 15, False), ("c128", 13, True)])
@pytest.mark.parametrize("circuit", [low_two_qubit, diagonals])
def test_pass_kernels(qs, circuit, dtype, n, fp64, policy):
    gates = circuit(n, qi.rng(17 * n), dtype == "c64")
    psi = qi.random_state(n, n)
    want = oracle.apply_circuit(psi.copy(), n, gates)
    qs.jit_set_policy(policy)
    before = qs.jit_stats()
    got = qs.State(n, dtype=dtype).set(psi).apply(gates, mode="tiled", fp64=fp64).get()
    after = qs.jit_stats()
    assert after["failed"] == before["failed"]
    if policy == "sync":  # every pass ran on its specialised kernel
        assert after["generic_launches"] == before["generic_launches"]
        assert after["specialised_launches"] > before["specialised_launches"]
    mx, l2 = TOL[dtype]
    assert np.max(np.abs(got - want)) <= mx and np.linalg.norm(got - want) <= l2


@pytest.mark.parametrize("n", [5, 12, 14])
def test_low_swaps_of_complex128_are_exact(qs, n):
    gates = [qi.Gate("SWAP", (n - 1, n - 4)), qi.Gate("SWAP", (n - 2, n - 1))]
    psi = qi.random_state(n, 3) * 2.0 ** qi.rng(1).integers(-300, 1, size=1 << n)
    want = oracle.apply_circuit(psi.copy(), n, gates)
    got = qs.State(n, dtype="c128").set(psi).apply(gates).get()
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("n", [13, 20, 21])
def test_gradient_over_few_and_many_tiles(qs, n):
    """2, 256 and 512 tiles per member (complex64): the reduction's two forms,
    against parameter shifts of the energy (tolerance: the energies' rounding,
    2^-24 per gate on amplitudes, 2 sum|c|)."""
    import torch
    gates = qi.variational_circuit(n, np.zeros((2, n)))
    index, count = qs.param_indices(gates)
    terms = qi.tfim_terms(n, 0.9)
    eng = qs.EnergyGradient(n, 1, gates, index, terms)
    params = torch.from_numpy(qi.rng(n).uniform(0, 6.28, size=(1, count))).cuda()
    grad = eng.run(params)[1].cpu().numpy().copy()
    for j in (0, 7, 8, n, count - 1):
        e = []
        for sign in (1.0, -1.0):
            p = params.clone()
            p[:, j] += sign * np.pi / 2
            e.append(float(eng.run(p, mode="forward")[0].cpu()))
        assert abs((e[0] - e[1]) / 2 - grad[0, j]) <= 2 * sum(abs(t[0]) for t in terms) * len(gates) * 2.0 ** -24
