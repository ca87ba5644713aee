"""Which queues on states below a tile run in one launch: long ones on few
members do; one gate, and short queues on many members, have a launch per gate
(then the amplitudes are those of mode "unfused" bit by bit). Members by the
thousand in one launch agree with the one-gate kernels within 4 u per gate."""
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


def launches(qs, fn):
    """(launches of the multi-gate kernel, other launches)"""
    qs.profile_collect()
    qs.profile_enable(True)
    fn()
    qs.profile_enable(False)
    p = qs.profile_collect()
    return p["tiled"][1], sum(v[1] for k, v in p.items() if k != "tiled")


@pytest.mark.parametrize("dtype,n,batch,count,one", [
    ("c64", 4, 1, 1, False), ("c64", 4, 1, 3, False), ("c64", 4, 1, 4, True), ("c64", 10, 1, 150, True),
    ("c64", 9, 1, 1, False), ("c64", 12, 300, 1, False), ("c64", 2, 16384, 40, True), ("c64", 2, 16385, 40, False),
    ("c64", 8, 1024, 4, True), ("c64", 8, 1025, 4, False), ("c64", 10, 2048, 32, True), ("c64", 10, 2049, 32, False),
    ("c64", 12, 257, 4, False), ("c64", 12, 3000, 16, True), ("c64", 12, 3000, 15, False),
    ("c128", 3, 4096, 32, True), ("c128", 3, 4097, 32, False), ("c128", 9, 128, 4, True), ("c128", 9, 129, 4, False),
    ("c128", 11, 512, 32, True), ("c128", 11, 513, 32, False), ("c128", 2, 1, 2, False)])
def test_route_by_gates_and_members(qs, dtype, n, batch, count, one):
    gates = [qi.Gate("U3", (k % n,), (), (0.1 + k, 0.2, 0.3)) for k in range(count)]
    psi = np.stack([qi.random_state(n, 7 + b) for b in range(min(batch, 5))])
    psi = np.concatenate([psi] * (batch // len(psi) + 1))[:batch]
    a, b = qs.State(n, batch=batch, dtype=dtype).set(psi), qs.State(n, batch=batch, dtype=dtype).set(psi)
    assert launches(qs, lambda: a.apply(gates)) == ((1, 0) if one else (0, count))
    x, y = a.get(), b.apply(gates, mode="unfused").get()
    if one:
        assert np.max(np.abs(x - y)) <= 4 * UNIT[dtype] * count * np.max(np.abs(y))
    else:
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("dtype,n,batch,layers,one", [
    ("c64", 2, 3072, 1, True), ("c64", 2, 3073, 1, False), ("c64", 1, 1, 1, False), ("c64", 10, 4096, 4, True),
    ("c64", 10, 4097, 4, False), ("c64", 11, 5000, 1, True), ("c128", 5, 9217, 1, False), ("c128", 6, 9217, 1, True)])
def test_route_of_member_angles(qs, dtype, n, batch, layers, one):
    import torch
    gates = []
    for layer in range(layers):
        gates += [qi.Gate("RY", (q,), (), (0.1,)) for q in range(n)]
        gates += [qi.Gate("CZ", (q, q + 1)) for q in range(n - 1)]
    index, count = qs.param_indices(gates)
    params = torch.from_numpy(qi.rng(n).uniform(0, 6.28, size=(batch, count))).cuda()
    a, b = qs.State(n, batch=batch, dtype=dtype).init_plus(), qs.State(n, batch=batch, dtype=dtype).init_plus()
    assert launches(qs, lambda: a.apply_batched(gates, index, params)) == ((1, 0) if one else (0, len(gates)))
    x, y = a.get(), b.apply_batched(gates, index, params, mode="unfused").get()
    assert np.max(np.abs(x - y)) <= 4 * UNIT[dtype] * len(gates) * np.max(np.abs(y))
