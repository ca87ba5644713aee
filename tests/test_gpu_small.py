"""GPU parity of gate queues on states below a tile, which run in one launch:
the one-gate kernels (mode "unfused") do the same arithmetic in the same order,
so the amplitudes agree to the last rounding of a fused multiply-add: within
4 u per gate of the state's largest amplitude (u = 2^-24 complex64, 2^-46 for
the double-float gates of complex128). Sizes 1 to 12 qubits (the last of each
precision is the largest below a tile), queues longer than a launch holds
(gates, matrix entries, per-member angles, gradient ops), 4-target unitaries
between them, batches, and complex128 in FP64. Gradients of queues that take
several launches against parameter shifts of the energy (tolerance: the
energies' own, 2 sum|c| * 4 u per gate)."""
import numpy as np
import pytest

from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu

UNIT = {"c128": 2.0 ** -46, "c64": 2.0 ** -24}


@pytest.fixture(scope="module")
def qs():
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    return qsim


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("dtype,n,batch,count", [
    ("c64", 1, 3, 40), ("c64", 2, 1, 60), ("c64", 5, 2, 1200), ("c64", 9, 1, 100), ("c64", 12, 2, 300),
    ("c128", 1, 3, 40), ("c128", 2, 1, 60), ("c128", 5, 2, 1200), ("c128", 9, 1, 100), ("c128", 11, 2, 300)])
def test_queue_matches_one_gate_kernels(qs, dtype, n, batch, count, fp64):
    if fp64 and dtype == "c64":
        pytest.skip("complex64 has one arithmetic")
    gates = qi.random_mixed_circuit(n, count, seed=n, max_unitary_k=4)
    psi = np.stack([qi.random_state(n, 90 + b) for b in range(batch)])
    a = qs.State(n, batch=batch, dtype=dtype).set(psi).apply(gates, fp64=fp64).get()
    b = qs.State(n, batch=batch, dtype=dtype).set(psi).apply(gates, mode="unfused", fp64=fp64).get()
    assert np.max(np.abs(a - b)) <= 4 * UNIT[dtype] * count * np.max(np.abs(b))


@pytest.mark.parametrize("dtype,n", [("c64", 3), ("c64", 12), ("c128", 3), ("c128", 11)])
def test_member_angles(qs, dtype, n):
    import torch
    B, r = 3, qi.rng(n)
    gates, index = [], []
    for k in range(300):  # more per-member angles than a launch holds
        kind = ("RX", "RY", "RZ", "U1", "CU1")[k % 5]
        q = [int(x) for x in r.permutation(n)]
        w = 2 if kind == "CU1" else 1
        gates.append(qi.Gate(kind, tuple(q[:w]), tuple(q[w:w + (k % 2)]), (0.0,)))
        index.append(k % 40)
    params = torch.from_numpy(r.uniform(0, 6.28, size=(B, 40))).cuda()
    psi = np.stack([qi.random_state(n, 60 + b) for b in range(B)])
    a = qs.State(n, batch=B, dtype=dtype).set(psi).apply_batched(gates, index, params).get()
    b = qs.State(n, batch=B, dtype=dtype).set(psi).apply_batched(gates, index, params, mode="unfused").get()
    assert np.max(np.abs(a - b)) <= 4 * UNIT[dtype] * 300 * np.max(np.abs(b))


@pytest.mark.parametrize("dtype,n", [("c64", 4), ("c64", 11), ("c128", 4), ("c128", 10)])
def test_gradients_over_several_launches(qs, dtype, n):
    import torch
    B, r = 2, qi.rng(3 * n)
    gates = []
    for k in range(130):  # more gradient ops than a launch holds
        q = [int(x) for x in r.permutation(n)]
        gates.append(qi.Gate(("RX", "RY", "RZ", "U1")[k % 4], (q[0],), (), (0.0,)))
        gates.append(qi.Gate("CZ", (q[1], q[2])))
    index, count = qs.param_indices(gates)
    terms = qi.tfim_terms(n, 0.7)
    eng = qs.EnergyGradient(n, B, gates, index, terms, dtype=dtype)
    params = torch.from_numpy(r.uniform(0, 6.28, size=(B, count))).cuda()
    energy, grad = (t.cpu().numpy().copy() for t in eng.run(params))
    tol = 2 * sum(abs(t[0]) for t in terms) * 4 * UNIT[dtype] * len(gates)
    for j in (0, 1, 2, 63, 64, 65, 127, 128):  # +-pi/2: exact for a rotation or phase without controls
        e = []
        for sign in (1.0, -1.0):
            p = params.clone()
            p[:, j] += sign * np.pi / 2
            e.append(eng.run(p, mode="forward")[0].cpu().numpy())
        assert np.max(np.abs((e[0] - e[1]) / 2 - grad[:, j])) <= tol
