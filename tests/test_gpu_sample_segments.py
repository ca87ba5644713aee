"""Samples of a walk that starts at a segment are those of the whole walk: n = 11
has no segments, and a 12-qubit state that holds the same amplitudes in one half
and zeros in the other has the same sums."""
import numpy as np
import pytest

from paper_2009_01845_gb300 import inputs as qi
from test_gpu_measure_walk import states

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("kind", [0, 2, 3])  # 1, the sparse one, has no amplitude left at n = 11
def test_segment_start_gives_the_whole_walks_samples(dtype, kind):
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    n = 11
    psi = states(n)[kind]
    u = np.concatenate([[0.0, 2.0 ** -53, 0.5, 1 - 2.0 ** -53], qi.rng(kind).uniform(size=200000)])
    want = qsim.State(n, dtype=dtype).set(psi).sample(u)
    zero = np.zeros_like(psi)
    low = qsim.State(n + 1, dtype=dtype).set(np.concatenate([psi, zero])).sample(u)
    high = qsim.State(n + 1, dtype=dtype).set(np.concatenate([zero, psi])).sample(u)
    np.testing.assert_array_equal(low, want)
    np.testing.assert_array_equal(high, want + (1 << n))


@pytest.mark.parametrize("kind", ["dense", "sparse", "spread"])
def test_few_shots_are_those_of_many(kind):
    """complex128 at n = 26: fewer than 2048 shots walk their blocks from the start."""
    import torch
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    n = 26
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn(1 << n, dtype=torch.complex128, device="cuda", generator=g)
    w = torch.rand(1 << n, dtype=torch.float64, device="cuda", generator=g)
    if kind == "sparse":
        psi[w > 1e-4] = 0
    elif kind == "spread":
        psi *= 10.0 ** (-12 * w)
    st = qsim.State(n, dtype="c128", tensor=psi)
    u = torch.from_numpy(np.concatenate([[0.0, 2.0 ** -53, 0.5, 1 - 2.0 ** -53], qi.rng(n).uniform(size=4092)])).cuda()
    apart = torch.cat([st.sample(c) for c in u.split(512)])
    assert torch.equal(apart, st.sample(u))
