"""Routes of dense 2-qubit gates and SWAPs on the low index bits: alone where a
pass would hold nothing else and a launch each moves less, in a tiled pass
beside other gates; complex128 in FP64 keeps the dense ones alone. Amplitudes
against the one-gate kernels, 4 u per gate of the largest."""
import numpy as np
import pytest

from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu

UNIT = {"c128": 2.0 ** -53, "c64": 2.0 ** -24}


def queue(name, n):
    r = qi.rng(n)
    q = lambda bit: n - 1 - bit  # noqa: E731
    u = lambda *t, c=(): qi.Gate("UNITARY", t, c, (), qi.random_unitary(2, r))  # noqa: E731
    return {"dense": [u(q(0), q(3))], "swap": [qi.Gate("SWAP", (q(1), 0))],
            "controlled": [u(q(k), q(9), c=(q(10), q(11))) for k in range(4)],
            "two": [u(q(0), 1), u(q(1), 2)], "beside": [u(q(0), q(3)), qi.Gate("U3", (q(7),), (), (0.1, 0.2, 0.3))],
            "swaps": [qi.Gate("SWAP", (k, q(k))) for k in range(6)]}[name]


@pytest.mark.parametrize("dtype,n,name,tiled", [
    ("c64", 14, "dense", 0), ("c64", 14, "two", 0), ("c64", 14, "swap", 0), ("c64", 14, "beside", 1),
    ("c64", 14, "swaps", 1), ("c64", 24, "dense", 0), ("c64", 24, "swap", 0), ("c64", 24, "controlled", 0),
    ("c64", 24, "two", 1), ("c64", 24, "beside", 1), ("c128", 13, "dense", 0), ("c128", 13, "beside", 1),
    ("c128", 13, "swap", 0), ("c128", 13, "swaps", 1)])
def test_route(dtype, n, name, tiled):
    from paper_2009_01845_gb300 import qsim as qs
    qs.load(build_if_missing=True)
    gates = queue(name, n)
    psi = qi.random_state(n, 1)
    st = qs.State(n, dtype=dtype).set(psi)
    qs.profile_collect()
    qs.profile_enable(True)
    st.apply(gates, fp64=True)
    qs.profile_enable(False)
    p = qs.profile_collect()
    alone = len(gates) if not tiled else 1 if (name, dtype) == ("beside", "c128") else 0
    assert p["tiled"][1] == tiled and sum(v[1] for k, v in p.items() if k != "tiled") == alone
    want = qs.State(n, dtype=dtype).set(psi).apply(gates, mode="unfused", fp64=True).get()
    assert np.max(np.abs(st.get() - want)) <= 4 * UNIT[dtype] * len(gates) * np.max(np.abs(want))
