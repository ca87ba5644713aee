"""The planner's cap on 2-qubit gates of the low index bits (CPU, emulated
passes): 24 of them take two passes, 24 whose low bit is only a control take one."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2009_01845_gb300 import inputs as qi
from paper_2009_01845_gb300 import qsim
from test_planner_emulated import TOL, emu  # noqa: F401 (fixture)


@pytest.mark.parametrize("dtype,low_target,passes", [(0, False, 1), (1, False, 1), (0, True, 2)])
def test_cap_counts_targets(emu, dtype, low_target, passes):  # noqa: F811
    n, r = 13, qi.rng(3)
    q = lambda bit: n - 1 - bit  # noqa: E731
    gates = []
    for k in range(24):
        if low_target:
            gates.append(qi.Gate("UNITARY", (q(7), q(k % 5)), (), (), qi.random_unitary(2, r)))
        else:
            gates.append(qi.Gate("UNITARY", (q(7), q(8)), (q(k % 5),), (), qi.random_unitary(2, r)))
    psi0 = qi.random_state(n, 1)
    psi = np.array(psi0, dtype=np.complex128)
    arr, keep = qsim.marshal_gates(gates)
    count = ctypes.c_int()
    assert emu.emu_apply_schedule(n, dtype, arr, len(gates), psi.ctypes.data, 0, 0, ctypes.byref(count)) == 0
    del keep
    assert np.max(np.abs(psi - oracle.run_circuit(n, gates, psi0))) < TOL[dtype]
    assert count.value == passes


@pytest.mark.parametrize("count,passes", [(1, 0), (2, 0), (5, 0), (6, 1)])
@pytest.mark.parametrize("kind", ["SWAP", "UNITARY"])
def test_few_alone_run_one_by_one(emu, kind, count, passes):  # noqa: F811
    n, r = 14, qi.rng(4)
    gates = [qi.Gate(kind, (n - 1 - k % 5, k), (7,) if k % 2 else (),
                     (), qi.random_unitary(2, r) if kind == "UNITARY" else None) for k in range(count)]
    psi0 = qi.random_state(n, 2)
    psi = np.array(psi0, dtype=np.complex128)
    arr, keep = qsim.marshal_gates(gates)
    ran = ctypes.c_int()
    assert emu.emu_apply_schedule(n, 0, arr, len(gates), psi.ctypes.data, 0, 0, ctypes.byref(ran)) == 0
    del keep
    assert np.max(np.abs(psi - oracle.run_circuit(n, gates, psi0))) < TOL[0]
    assert ran.value == passes
