"""H psi with many Z strings of weight above 2, which take tiles of 8 (complex128)
and 16 (complex64) outputs per thread: the sizes at which those begin, one size
below, states of one tile, batches, and large complex128 states without any. (A constant H is given as H0 = H1, whose terms
are added up: twice the strings.) Reference: the solver in NumPy complex128, L2
<= 64 u (see test_gpu_hpsi.py)."""
import numpy as np
import pytest

from paper_2009_01845_gb300 import inputs as qi
from test_gpu_hpsi import close, rk4

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n,batch,strings", [
    ("c64", 12, 128, 50), ("c64", 12, 128, 49), ("c64", 12, 127, 60), ("c64", 19, 1, 50), ("c64", 13, 65, 150),
    ("c128", 16, 1, 80), ("c128", 16, 1, 79), ("c128", 11, 64, 20), ("c128", 11, 64, 19), ("c128", 18, 1, 5),
    ("c128", 18, 1, 4), ("c128", 13, 64, 3), ("c128", 12, 17, 150),
    ("c128", 19, 1, 0), ("c128", 11, 1024, 0)])
def test_many_strings(dtype, n, batch, strings):
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    r = qi.rng(n + strings)
    h = [(-0.5, 1 << q, 0) for q in range(n)] + qi.random_ising_terms(n, r)[:20]
    if strings:
        h += [(0.3, 3, 5), (0.2, 1 << (n - 1), 1)]
    h += [(float(r.normal()) / 8, 0, sum(1 << int(b) for b in r.permutation(n)[:3 + k % 4])) for k in range(strings)]
    s = sum(abs(x[0]) for x in h)
    h = [(c / s, x, z) for c, x, z in h]
    psi = np.stack([qi.random_state(n, b) for b in range(min(batch, 3))])
    st = qsim.State(n, batch=batch, dtype=dtype).set(np.concatenate([psi] * (batch // len(psi) + 1))[:batch])
    psi = st.get().reshape(batch, -1)[:len(psi)].astype(np.complex128)
    got = st.evolve(h, h, 1.0, 1.0, solver="rk4").get().reshape(batch, -1)
    want = rk4(psi, n, h, 1.0)
    for b in range(batch):
        close(got[b], want[b % len(psi)], dtype)
