"""Queues on small complex128 states with the FP64 flag stay in FP64 in one
launch: within 4 u per gate of the one-gate FP64 kernels (u = 2^-53), also where
the amplitudes (2^-300) lie far below what a pair of floats can hold."""
import numpy as np
import pytest

from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch,count", [(2, 1, 60), (5, 2, 400), (9, 1, 100), (11, 2, 200)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300])
def test_queue_stays_in_fp64(n, batch, count, scale):
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    gates = qi.random_mixed_circuit(n, count, seed=n, max_unitary_k=3)
    psi = scale * np.stack([qi.random_state(n, 30 + b) for b in range(batch)])
    qsim.profile_collect()
    qsim.profile_enable(True)
    a = qsim.State(n, batch=batch, dtype="c128").set(psi).apply(gates, fp64=True).get()
    qsim.profile_enable(False)
    assert qsim.profile_collect()["tiled"][1] >= 1  # not a launch per gate
    b = qsim.State(n, batch=batch, dtype="c128").set(psi).apply(gates, mode="unfused", fp64=True).get()
    assert np.max(np.abs(b)) > 0.01 * scale / 2 ** (n / 2)
    assert np.max(np.abs(a - b)) <= 4 * 2.0 ** -53 * count * np.max(np.abs(b))
