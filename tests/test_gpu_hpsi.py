"""GPU parity of H psi (through the exact solvers, whose steps are applications
of H with their combinations): every kernel shape and its edges, in both
precisions (one output per thread below a tile; small, middle and large
tiles), every kind of term (transverse fields with one and with several
coefficients, strings with real and imaginary coefficients inside and outside
the tile and on its chunk bits, several strings on one X mask, Z strings of
weight 0 to 5), sums that take several launches, and batches.

Reference: the same solver in NumPy complex128. Tolerance: L2 <= 64 u with u
the unit roundoff of the arithmetic (2^-24 complex64, 2^-46 complex128 in
double-float), for dt sum|c| of about 1."""
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


def apply_h(psi, n, terms):
    x = np.arange(1 << n, dtype=np.int64)
    out = np.zeros_like(psi)
    rev = lambda m: sum(1 << (n - 1 - q) for q in range(n) if (m >> q) & 1)  # noqa: E731
    for c, xm, zm in terms:
        y = x ^ rev(xm)
        odd = np.bitwise_count(y & rev(zm)) & 1
        out += (c * 1j ** bin(xm & zm).count("1")) * np.where(odd, -1.0, 1.0) * psi[..., y]
    return out


def rk4(psi, n, h, dt):
    f = lambda v: -1j * apply_h(v, n, h)  # noqa: E731
    a = f(psi)
    b = f(psi + dt / 2 * a)
    c = f(psi + dt / 2 * b)
    return psi + dt / 6 * (a + 2 * b + 2 * c + f(psi + dt * c))


def taylor(psi, n, h, dt):
    term, out = psi.copy(), psi.copy()
    for j in range(1, 30):
        term = -1j * dt / j * apply_h(term, n, h)
        out = out + term
    return out


def terms_for(n, seed, strings):
    r = qi.rng(seed)
    t = [(-1.0, 1 << q, 0) for q in range(n) if q % 4]                  # one coefficient
    t += [(float(r.normal()), 1 << q, 0) for q in range(0, n, 4)]       # others
    t += qi.random_pauli_terms(n, strings, seed + 1)
    t += [(0.3, 1, 1 << (n - 1)), (-0.2, 1, 1), (0.1, 1, 3)]            # one X mask, several strings
    t += [(float(r.normal()), 0, (1 << i) | (1 << j)) for i in range(n) for j in range(i + 1, min(n, i + 4))]
    t += [(float(r.normal()), 0, 1 << i) for i in range(n)] + [(0.25, 0, 0)]
    t += [(float(r.normal()), 0, int(sum(1 << q for q in r.permutation(n)[:w]))) for w in (3, 4, 5) if n >= w]
    s = sum(abs(x[0]) for x in t)
    return [(c / s, x, z) for c, x, z in t]


def close(got, want, dtype):
    assert np.linalg.norm(got.reshape(want.shape).astype(np.complex128) - want) <= 64 * UNIT[dtype] * \
        np.linalg.norm(want)


@pytest.mark.parametrize("dtype,n,batch", [
    ("c64", 3, 2), ("c64", 7, 1), ("c64", 8, 3), ("c64", 9, 1), ("c64", 11, 1), ("c64", 10, 256), ("c64", 18, 1),
    ("c64", 12, 256), ("c64", 21, 1),
    ("c128", 3, 2), ("c128", 10, 1), ("c128", 11, 2), ("c128", 13, 1), ("c128", 11, 256), ("c128", 19, 1),
    ("c128", 11, 1024), ("c128", 20, 1)])
def test_h_psi_every_shape(qs, dtype, n, batch):
    h = terms_for(n, n, 12 if n < 20 else 8)
    psi = np.stack([qi.random_state(n, 7 * n + b) for b in range(batch)])
    st = qs.State(n, batch=batch, dtype=dtype).set(psi)
    psi = st.get().reshape(batch, -1).astype(np.complex128)
    # H0 = H1: a constant H; one step of dt = 1 in units of 1 / sum|c|
    close(st.evolve(h, h, 1.0, 1.0, solver="rk4").get(), rk4(psi, n, h, 1.0), dtype)


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("solver", ["exp", "rk4", "rk45"])
def test_sums_of_several_launches(qs, dtype, solver):
    n = 11
    h = terms_for(n, 3, 300)
    psi = qi.random_state(n, 5)
    st = qs.State(n, dtype=dtype).set(psi)
    psi = st.get().astype(np.complex128)
    if solver == "rk45":  # fifth order: at dt = 0.01 its error is below the tolerances
        want, T, dt = taylor(psi, n, h, 0.01), 0.01, 0.01
    elif solver == "rk4":
        want, T, dt = rk4(psi, n, h, 1.0), 1.0, 1.0
    else:
        want, T, dt = taylor(psi, n, h, 1.0), 1.0, 1.0
    close(st.evolve(h, h, T, dt, solver=solver).get(), want, dtype)
