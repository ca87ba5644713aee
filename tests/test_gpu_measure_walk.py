"""GPU parity of the measurement kernels at the edges of their fast forms: groups
that leave exactly 4, or only 3, index bits above the low 8 free (the register
bits of the marginal walk), and samples from states whose blocks of 4096 and
segments of 128 amplitudes are partly empty, hold one outcome, or span many
magnitudes (a shot starts its walk at a segment).

Tolerances: marginals 1e-12 (complex128) and 1e-6 (complex64), as 64-term runs
in the state's precision allow; a sample is right where its target lies within
the sums' rounding of its interval of the cumulative sum: 2e-6 for complex64
(16-term sums of rounded squares in FP32, 20 roundings of 2^-24), 1e-9 for
complex128."""
import numpy as np
import pytest

import oracle
from paper_2009_01845_gb300 import inputs as qi

pytestmark = pytest.mark.gpu

MTOL = {"c128": 1e-12, "c64": 1e-6}
STOL = {"c128": 1e-9, "c64": 2e-6}


@pytest.fixture(scope="module")
def qs():
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    return qsim


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,bits,batch", [
    (12, (0, 4, 7), 1), (12, (0, 1, 2, 3, 4), 3), (12, (8,), 1), (13, (12, 3), 2), (13, (8, 0), 1), (14, (8, 9), 1),
    (16, (8, 9, 10, 11), 2), (16, (15, 14, 13, 12, 11), 1), (20, (8, 10, 12, 14, 16, 18, 0, 1, 2, 3, 4, 7), 1),
    (20, (19, 18, 17, 16, 15, 14, 13, 12), 2), (18, (5, 6, 7), 1)])
def test_marginal_walk(qs, dtype, n, bits, batch):
    psi = np.stack([qi.random_state(n, 11 * n + b) for b in range(batch)])
    st = qs.State(n, batch=batch, dtype=dtype).set(psi)
    held = st.get().reshape(batch, -1).astype(np.complex128)
    group = [n - 1 - b for b in bits]
    got = st.marginal_probabilities(group).reshape(batch, -1)
    for b in range(batch):
        want = oracle.marginal_probabilities(np.ascontiguousarray(held[b]), n, group)
        assert np.max(np.abs(got[b] - want)) <= MTOL[dtype]


def states(n):
    r = qi.rng(n)
    dense = qi.random_state(n, n)
    sparse = np.where(r.uniform(size=1 << n) < 2e-3, dense, 0)
    sparse[(1 << n) // 2: (1 << n) // 2 + 4096] = 0
    spread = dense * 10.0 ** r.uniform(-12, 0, size=1 << n)
    ends = np.zeros(1 << n, dtype=complex)
    ends[127::128] = dense[127::128]            # the last amplitude of every segment
    ends[5000 % (1 << n):6000 % (1 << n)] = 0
    return [dense, sparse, spread, ends]


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n", [11, 12, 13, 17])
def test_sample_walk(qs, dtype, n):
    for i, psi0 in enumerate(states(n)):
        if not np.any(psi0):
            continue  # a zero vector is no state (the sparse one can be, at n = 11)
        st = qs.State(n, dtype=dtype).set(psi0 / np.linalg.norm(psi0))
        psi = np.ascontiguousarray(st.get().astype(np.complex128))
        cdf = np.cumsum(np.abs(psi) ** 2)
        # uniforms all over, and just around every 64th boundary
        edge = cdf[:: max(1, (1 << n) // 64)] / cdf[-1]
        u = np.concatenate([qi.rng(i).uniform(size=30000), edge - 3e-9, edge + 3e-9, [0.0, np.nextafter(1.0, 0.0)]])
        u = u[(u >= 0) & (u < 1)]
        got = st.sample(u).astype(np.int64)
        want = oracle.sample(psi, n, u).astype(np.int64)
        assert np.all(np.abs(psi[got]) > 0)
        bad = np.flatnonzero(got != want)
        target = u[bad] * cdf[-1]
        below = np.where(got[bad] > 0, cdf[np.maximum(got[bad] - 1, 0)], 0.0)
        assert np.all(below <= target + STOL[dtype]) and np.all(cdf[got[bad]] > target - STOL[dtype])
