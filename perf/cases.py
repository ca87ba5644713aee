"""The work a program has this framework do, as cases that can be timed and checked.

Every case goes through the public binding (``paper_2009_01845_gb300.qsim``): circuits as execution
plans and as one-off gate queues, energies with their gradients, adiabatic (Trotter) evolution of
several instances, the exact solvers, read-outs of a final state, and density matrices with noise.
A circuit that is run many times (a plan, a variational ansatz, a noisy circuit) is part of the case;
the seed draws what a program changes from run to run: the input state, the angles, the couplings, the
uniforms of the samples. Energies, gradients and probabilities of a complex64 simulation are kept in 32
bits, as a program that simulates in complex64 keeps them.
"""
import functools
import math

import numpy as np
import torch

from paper_2009_01845_gb300 import inputs as qi
from paper_2009_01845_gb300 import qsim

TDT = {"c64": torch.complex64, "c128": torch.complex128}
AMP = {"c64": 8, "c128": 16}
C128 = torch.complex128


def listed():
    return [
        # a small circuit of mixed gates run again and again from a plan (test and teaching sizes,
        # the inner circuit of a hybrid program): latency of one execution
        {"name": "mixed_plan_c64_n10", "kind": "plan", "circuit": "mixed", "n": 10, "size": 150, "dtype": "c64"},
        # the quantum Fourier transform of a basis state, as the paper times it, in double precision
        {"name": "qft_plan_c128_n18", "kind": "plan", "circuit": "qft", "n": 18, "size": 0, "dtype": "c128"},
        # the headline circuit family: 20 random layers, at the largest size that can be checked here
        {"name": "layers_plan_c64_n28", "kind": "plan", "circuit": "layers", "n": 28, "size": 20, "dtype": "c64"},
        # the same family in double precision
        {"name": "layers_plan_c128_n25", "kind": "plan", "circuit": "layers", "n": 25, "size": 10, "dtype": "c128"},
        # a circuit that is run once (a compiled program with controls, swaps and 3-qubit unitaries):
        # planning and the kernels that need no preparation
        {"name": "mixed_once_c64_n23", "kind": "once", "circuit": "mixed", "n": 23, "size": 60, "dtype": "c64"},
        # training step of the hardware-efficient ansatz over a batch of parameter sets: energy of the
        # transverse-field Ising chain and its gradient
        {"name": "gradient_c64_n18_b64", "kind": "gradient", "n": 18, "batch": 64, "layers": 10, "dtype": "c64"},
        # the same at the size of a small chemistry or teaching problem, in double precision
        {"name": "gradient_c128_n10_b8", "kind": "gradient", "n": 10, "batch": 8, "layers": 4, "dtype": "c128"},
        # adiabatic optimisation of random Ising instances of several widths in one call
        {"name": "adiabatic_c64_n16_22", "kind": "adiabatic", "n_lo": 16, "n_hi": 22, "count": 16, "steps": 20,
         "dtype": "c64"},
        # exact time evolution by Runge-Kutta: dense Ising couplings plus random Pauli strings
        {"name": "rk4_c64_n24", "kind": "evolve", "solver": "rk4", "n": 24, "steps": 4, "dtype": "c64"},
        # the exponential solver at the size of a reference calculation, in double precision
        {"name": "exp_c128_n16", "kind": "evolve", "solver": "exp", "n": 16, "steps": 3, "dtype": "c128"},
        # read-outs of one final state: energy, norm, a register's outcome probabilities, samples
        {"name": "readout_c64_n27", "kind": "readout", "n": 27, "group": 8, "shots": 100000, "dtype": "c64"},
        # a noisy circuit on a density matrix: random layers, each followed by depolarizing channels
        {"name": "noisy_density_c64_n13", "kind": "density", "n": 13, "layers": 2, "dtype": "c64"},
    ]


def draw(rng):
    """One more case of the listed ranges."""
    def spread(lo, hi):  # over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plan", "plan", "plan", "once", "gradient", "adiabatic", "evolve", "readout", "density"])
    dtype = rng.choice(["c64", "c64", "c128"])
    if kind == "plan":
        circuit = rng.choice(["mixed", "qft", "layers"])
        n = {"mixed": rng.randint(3, 16), "qft": rng.randint(4, 24),
             "layers": rng.randint(14, 27 if dtype == "c64" else 24)}[circuit]
        size = {"mixed": spread(20, 200), "qft": 0, "layers": rng.randint(2, 12)}[circuit]
        return {"kind": kind, "circuit": circuit, "n": n, "size": size, "dtype": dtype}
    if kind == "once":
        circuit = rng.choice(["mixed", "layers"])
        return {"kind": kind, "circuit": circuit, "n": rng.randint(9, 23),
                "size": rng.randint(2, 60) if circuit == "mixed" else rng.randint(1, 8), "dtype": dtype}
    if kind == "gradient":
        n = rng.randint(4, 18)
        return {"kind": kind, "n": n, "batch": spread(1, min(256, 1 << (22 - n))), "layers": rng.randint(1, 10),
                "dtype": dtype}
    if kind == "adiabatic":
        lo = rng.randint(13, 20)
        return {"kind": kind, "n_lo": lo, "n_hi": min(22, lo + rng.randint(0, 5)), "count": rng.randint(1, 16),
                "steps": rng.randint(3, 20), "dtype": dtype}
    if kind == "evolve":
        return {"kind": kind, "solver": rng.choice(["exp", "rk4", "rk45"]), "n": rng.randint(6, 21),
                "steps": rng.randint(1, 4), "dtype": dtype}
    if kind == "readout":
        n = rng.randint(11, 27 if dtype == "c64" else 25)
        return {"kind": kind, "n": n, "group": rng.randint(1, 11), "shots": spread(100, 200000), "dtype": dtype}
    return {"kind": kind, "n": rng.randint(4, 13 if dtype == "c64" else 12), "layers": rng.randint(1, 2),
            "dtype": dtype}


# ------------------------------------------------------------------ what a program has in hand
@functools.lru_cache(maxsize=64)
def gates_of(circuit, n, size, seed):
    """size: the gates of a mixed circuit, the layers of random layers."""
    if circuit == "qft":
        return qi.qft_circuit(n)
    if circuit == "layers":
        return qi.random_layer_circuit(n, size, seed=seed)
    return qi.random_mixed_circuit(n, size, seed=seed, max_controls=2, max_unitary_k=3)


def circuit_of(c, seed):
    """The case's circuit: a plan's is its own, a one-off queue's is drawn from the seed."""
    return gates_of(c["circuit"], c["n"], c["size"], 2 if c["kind"] == "plan" else 1000 + seed)


def basis_of(c, seed):
    return int(qi.rng(seed).integers(0, 1 << c["n"]))


def random_state(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    v = torch.randn(1 << n, dtype=TDT[dtype], device="cuda", generator=g)
    return v.div_(torch.linalg.vector_norm(v))


def final_state(n, dtype, seed):
    """A state like those at the end of a run, with an energy of the order of its terms: a product of one-qubit
    states plus noise."""
    r = qi.rng(seed)
    v = torch.ones(1, dtype=C128, device="cuda")
    for _ in range(n):
        t, f = r.uniform(0.3, 1.2), r.uniform(-0.6, 0.6)
        q = torch.tensor([math.cos(t), math.sin(t) * complex(math.cos(f), math.sin(f))], dtype=C128, device="cuda")
        v = (v[:, None] * q[None, :]).reshape(-1)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    w = torch.randn(1 << n, dtype=TDT[dtype], device="cuda", generator=g)
    v += w * (0.3 * 2.0 ** (-n / 2))
    del w
    return (v / torch.linalg.vector_norm(v)).to(TDT[dtype])


def ansatz(c):
    gates = qi.variational_circuit(c["n"], np.zeros((c["layers"], c["n"])))
    index, count = qsim.param_indices(gates)
    return gates, index, count


def angles(c, seed):
    t = qi.variational_params(c["batch"], c["layers"], c["n"], seed=seed)
    return torch.from_numpy(t.reshape(c["batch"], -1)).cuda()


def instances(c, seed):
    """The widths of the case and, per width, its instances' H1 (drawn from the seed)."""
    r = qi.rng(seed)
    span = c["n_hi"] - c["n_lo"] + 1
    widths = [c["n_lo"] + i * span // c["count"] for i in range(c["count"])]
    by = {}
    for w in widths:
        by.setdefault(w, []).append(qi.random_ising_terms(w, r))
    return by


def hamiltonians(c, seed):
    n = c["n"]
    return qi.transverse_field_terms(n), qi.random_ising_terms(n, qi.rng(seed)) + qi.random_pauli_terms(n, 8, seed + 1)


def depolarizing(p=0.01):
    X = np.array([[0, 1], [1, 0]], dtype=complex)
    Y = np.array([[0, -1j], [1j, 0]], dtype=complex)
    Z = np.diag([1.0, -1.0]).astype(complex)
    return [math.sqrt(1 - 3 * p / 4) * np.eye(2), math.sqrt(p / 4) * X, math.sqrt(p / 4) * Y, math.sqrt(p / 4) * Z]


def noisy_layers(c):
    gates = gates_of("layers", c["n"], c["layers"], 6)
    per = [[] for _ in range(c["layers"])]
    layer, seen = -1, 0
    for g in gates:  # a layer is n U3 gates, then its CZ gates
        if g.kind == "U3":
            if seen % c["n"] == 0:
                layer += 1
            seen += 1
        per[layer].append(g)
    return per


DT = 0.01  # time step of the evolutions


class Box(dict):
    __getattr__ = dict.__getitem__


def prepare(case, seed):
    c, kind, dt = case, case["kind"], case["dtype"]
    s = Box(case=case)
    qsim.jit_set_policy("off" if kind == "once" else "tiered")
    if kind in ("plan", "once"):
        s["x"] = basis_of(c, seed)
        s["state"] = qsim.State(c["n"], dtype=dt).init_basis(s.x)
        s["gates"] = circuit_of(c, seed)
        if kind == "plan":
            s["plan"] = qsim.Plan(s.state, s.gates)
    elif kind == "gradient":
        gates, index, _ = ansatz(c)
        s["engine"] = qsim.EnergyGradient(c["n"], c["batch"], gates, index, qi.tfim_terms(c["n"], 1.0), dtype=dt)
        s["params"] = angles(c, seed)
    elif kind == "adiabatic":
        by = instances(c, seed)
        s["states"] = [qsim.State(w, batch=len(h), dtype=dt) for w, h in by.items()]
        s["h0"] = [qi.transverse_field_terms(w) for w in by]
        s["h1"] = [t for h in by.values() for t in h]
    elif kind == "evolve":
        s["psi0"] = random_state(c["n"], dt, seed)
        s["state"] = qsim.State(c["n"], dtype=dt)
        s["h0"], s["h1"] = hamiltonians(c, seed)
    elif kind == "readout":
        s["state"] = qsim.State(c["n"], dtype=dt, tensor=final_state(c["n"], dt, seed))
        s["terms"] = qi.tfim_terms(c["n"], 1.0)
        s["group"] = sorted(int(q) for q in qi.rng(c["n"]).permutation(c["n"])[:c["group"]])
        s["uniforms"] = torch.from_numpy(qi.rng(seed).uniform(size=c["shots"])).cuda()
    elif kind == "density":
        s["state"] = qsim.DensityMatrix(c["n"], dtype=dt)
        s["psi"] = qi.random_state(c["n"], seed)
        s["layers"] = noisy_layers(c)
        s["noise"] = [([q], depolarizing()) for q in range(c["n"])]
    else:
        raise ValueError(kind)
    if kind in ("gradient", "adiabatic", "density"):
        # a program that repeats these circuits has had their pass kernels specialised by its first runs
        qsim.jit_set_policy("eager")
        run(s)
        qsim.jit_wait()
        qsim.jit_set_policy("tiered")
    torch.cuda.synchronize()
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    single = c["dtype"] == "c64"
    if kind == "plan":
        s.state.init_basis(s.x)
        s.plan.execute()
        return s.state.tensor
    if kind == "once":
        return s.state.init_basis(s.x).apply(s.gates).tensor
    if kind == "gradient":
        energy, grad = s.engine.run(s.params)
        return [energy.float(), grad.float()] if single else [energy, grad]
    if kind == "adiabatic":
        for st in s.states:
            st.init_plus()
        qsim.adiabatic_run_batch(s.states, s.h0, s.h1, 1000 * DT, DT, steps=c["steps"])
        return [st.tensor for st in s.states]
    if kind == "evolve":
        s.state.set(s.psi0)
        s.state.evolve(s.h0, s.h1, c["steps"] * DT, DT, solver=c["solver"])
        return s.state.tensor
    if kind == "readout":
        real = np.float32 if single else np.float64
        st = s.state
        energy = st.expectation(s.terms).real.astype(real)
        norm = st.norm2().astype(real)
        probs = st.marginal_probabilities(s.group).astype(real)
        return [energy, norm, probs, st.sample(s.uniforms)]
    s.state.init_pure(s.psi)
    for gates in s.layers:
        s.state.apply(gates)
        s.state.apply_channels(s.noise)
    return s.state.tensor


# ------------------------------------------------------------------ what a pass cannot do without
def gate_flops(g):
    """Real operations per amplitude of the state: a complex 2^k x 2^k product, six for a phase, on the part of the
    amplitudes that the controls select."""
    part = 0.5 ** len(g.controls)
    if g.kind in ("Z", "S", "SDG", "T", "TDG", "U1"):
        return 6.0 * part / 2
    if g.kind in ("CZ", "CU1"):
        return 6.0 * part / 4
    if g.kind == "RZ":
        return 6.0 * part
    if g.kind in ("X", "SWAP"):
        return 0.0
    return (8.0 * 2 ** len(g.targets) - 2) * part


def work(case):
    c, kind = case, case["kind"]
    if kind in ("plan", "once"):
        amps = float(1 << c["n"])
        return {"bytes": amps * AMP[c["dtype"]], "flops": amps * sum(gate_flops(g) for g in circuit_of(c, 0))}
    if kind == "gradient":
        # forward: the ansatz on psi; backward: on psi and lambda, and one product per parameter; H psi
        n, params = c["n"], c["layers"] * c["n"]
        amps = float(c["batch"] << n)
        return {"bytes": 8.0 * c["batch"] * (2 * params + 1), "flops": amps * (3 * 6 * params + 4 * params + 4 * n)}
    if kind == "adiabatic":
        by = instances(c, 0)
        amps = {w: float(len(h) << w) for w, h in by.items()}
        # per step and amplitude: one phase, and one real rotation per qubit
        return {"bytes": sum(amps.values()) * AMP[c["dtype"]],
                "flops": c["steps"] * sum(a * (6 + 6 * w) for w, a in amps.items())}
    if kind == "evolve":
        amps = float(1 << c["n"])
        h = evolve_products(c)
        # each product with H reads one state and writes one; n + 8 partners are added up per amplitude
        return {"bytes": 2.0 * h * amps * AMP[c["dtype"]], "flops": h * amps * (2 * c["n"] + 8 * 8 + 4)}
    if kind == "readout":
        amps = float(1 << c["n"])
        return {"bytes": amps * AMP[c["dtype"]] + 16.0 * c["shots"], "flops": amps * (4 * c["n"] + 8)}
    amps = float(1 << (2 * c["n"]))
    flops = sum(2 * gate_flops(g) for layer in noisy_layers(c) for g in layer) + c["layers"] * c["n"] * 30.0
    return {"bytes": amps * AMP[c["dtype"]], "flops": amps * flops}


def evolve_products(c):
    """Products with H in one pass."""
    if c["solver"] != "exp":
        return c["steps"] * (4 if c["solver"] == "rk4" else 6)
    h0, h1 = hamiltonians(c, 0)
    total = 0
    for k in range(c["steps"]):
        H = mixed_terms(h0, h1, (k + 0.5) / c["steps"])
        nu = sum(abs(t[0]) for t in H)
        pieces = max(1, math.ceil(nu * DT))
        eps = 6e-8 if c["dtype"] == "c64" else 1.2e-16
        order, b = 1, nu * DT / pieces
        while order < 60:
            b *= nu * DT / pieces / (order + 1)
            if b <= eps:
                break
            order += 1
        total += pieces * order
    return total


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def matrix_of(g):
    if g.matrix is not None:
        return np.asarray(g.matrix, dtype=complex)
    p = list(g.params)
    s = 1 / math.sqrt(2)
    e = lambda a: complex(math.cos(a), math.sin(a))  # noqa: E731
    u3 = lambda t, f, l: np.array([[math.cos(t / 2), -e(l) * math.sin(t / 2)],  # noqa: E731, E741
                                   [e(f) * math.sin(t / 2), e(f + l) * math.cos(t / 2)]])
    k = g.kind
    if k == "H":
        return np.array([[s, s], [s, -s]], dtype=complex)
    if k == "X":
        return np.array([[0, 1], [1, 0]], dtype=complex)
    if k == "Y":
        return np.array([[0, -1j], [1j, 0]])
    if k in ("Z", "S", "SDG", "T", "TDG", "U1"):
        a = {"Z": math.pi, "S": math.pi / 2, "SDG": -math.pi / 2, "T": math.pi / 4, "TDG": -math.pi / 4}.get(k)
        return np.diag([1, e(p[0] if a is None else a)])
    if k == "RX":
        return np.array([[math.cos(p[0] / 2), -1j * math.sin(p[0] / 2)], [-1j * math.sin(p[0] / 2), math.cos(p[0] / 2)]])
    if k == "RY":
        return np.array([[math.cos(p[0] / 2), -math.sin(p[0] / 2)], [math.sin(p[0] / 2), math.cos(p[0] / 2)]], dtype=complex)
    if k == "RZ":
        return np.diag([e(-p[0] / 2), e(p[0] / 2)])
    if k == "U2":
        return u3(math.pi / 2, p[0], p[1])
    if k == "U3":
        return u3(*p)
    if k == "CZ":
        return np.diag([1, 1, 1, -1]).astype(complex)
    if k == "CU1":
        return np.diag([1, 1, 1, e(p[0])])
    if k == "SWAP":
        return np.array([[1, 0, 0, 0], [0, 0, 1, 0], [0, 1, 0, 0], [0, 0, 0, 1]], dtype=complex)
    raise ValueError(k)


def apply_matrix(psi, n, targets, controls, u):
    """u on the targets (the first is the local most significant bit) of the part of psi whose controls are 1."""
    where = sorted(list(targets) + list(controls))
    shape, last = [], -1
    for q in where:
        shape += [1 << (q - last - 1), 2]
        last = q
    v = psi.view(shape + [1 << (n - 1 - last)])

    def part(local):
        index = [slice(None)] * v.dim()
        for q in controls:
            index[2 * where.index(q) + 1] = 1
        for j, q in enumerate(targets):
            index[2 * where.index(q) + 1] = (local >> (len(targets) - 1 - j)) & 1
        return v[tuple(index)]

    d = 1 << len(targets)
    if not np.any(u - np.diag(np.diag(u))):
        for i in range(d):
            if u[i, i] != 1:
                part(i).mul_(complex(u[i, i]))
        return
    new = {}
    for i in range(d):
        row = None
        for j in range(d):
            if u[i, j] != 0:
                row = part(j) * complex(u[i, j]) if row is None else row.add_(part(j), alpha=complex(u[i, j]))
        new[i] = torch.zeros_like(part(i)) if row is None else row
    for i in range(d):
        part(i).copy_(new[i])


def signs(n, zmask):
    """(-1)^(number of mask qubits that are 1), as one float64 per basis index."""
    v = torch.ones(1, dtype=torch.float64, device="cuda")
    for q in range(n):
        z = torch.tensor([1.0, -1.0 if (zmask >> q) & 1 else 1.0], dtype=torch.float64, device="cuda")
        v = (v[:, None] * z[None, :]).reshape(-1)
    return v


class PauliSum:
    """A Pauli sum to be applied to a state: per X mask, the coefficient of every basis index. The terms of two sums
    with the same masks share the work."""

    def __init__(self, n, terms):
        self.n = n
        self.groups = {}
        bit = 1 << torch.arange(n - 1, -1, -1, device="cuda")
        self.index = torch.arange(1 << n, device="cuda")
        for coeff, xm, zm in terms:
            c = coeff * (1j ** bin(xm & zm).count("1"))
            if zm == 0:
                self.groups.setdefault(xm, [0, None])[0] += c
            else:
                g = self.groups.setdefault(xm, [0, None])
                part = signs(n, zm)
                # only a term with Y has a complex factor
                part = part * c if abs(complex(c).imag) else part * complex(c).real
                g[1] = part if g[1] is None else g[1] + part
        self.shift = {xm: int(sum(int(bit[q]) for q in range(n) if (xm >> q) & 1)) for xm in self.groups}

    def add(self, psi, out, scale):
        for xm, (const, var) in self.groups.items():
            src = psi
            if var is not None:
                src = psi * (var + const if const else var)
            if self.shift[xm]:
                src = src[self.index ^ self.shift[xm]]
            out.add_(src, alpha=complex(scale * (const if var is None else 1)))


def mixed_terms(h0, h1, s):
    return [((1 - s) * c, x, z) for c, x, z in h0] + [(s * c, x, z) for c, x, z in h1]


def exact_evolve(c, seed):
    n = c["n"]
    h0, h1 = hamiltonians(c, seed)
    P0, P1 = PauliSum(n, h0), PauliSum(n, h1)
    T = c["steps"] * DT
    y = random_state(n, c["dtype"], seed).to(C128)

    def f(t, v, scale=-1j):
        out = torch.zeros_like(v)
        P0.add(v, out, 1 - t / T)
        P1.add(v, out, t / T)
        return out.mul_(scale)

    if c["solver"] == "exp":
        for k in range(c["steps"]):
            t = (k + 0.5) * DT
            nu = sum(abs(x[0]) for x in mixed_terms(h0, h1, t / T))
            pieces = max(1, math.ceil(nu * DT))
            for _ in range(pieces):
                term = y.clone()
                for j in range(1, 26):
                    term = f(t, term, -1j * DT / pieces / j)
                    y += term
        return y
    if c["solver"] == "rk4":
        for k in range(c["steps"]):
            t = k * DT
            a = f(t, y)
            b = f(t + DT / 2, y + DT / 2 * a)
            d = f(t + DT / 2, y + DT / 2 * b)
            e = f(t + DT, y + DT * d)
            y = y + DT / 6 * (a + 2 * b + 2 * d + e)
        return y
    nodes = [0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1]
    A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
         [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
         [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656]]
    B = [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]
    for k in range(c["steps"]):
        ks = []
        for i in range(6):
            v = y.clone()
            for j, a in enumerate(A[i]):
                v += DT * a * ks[j]
            ks.append(f(k * DT + nodes[i] * DT, v))
        for b, kk in zip(B, ks):
            y = y + DT * b * kk
    return y


def exact_gradient(c, seed):
    n, B, L = c["n"], c["batch"], c["layers"]
    th = angles(c, seed).view(B, L, n)
    H = PauliSum(n, qi.tfim_terms(n, 1.0))

    def ry(v, q, t):  # in place on every member (rows of v may come in several states per member)
        w = v.view(B, -1, 1 << q, 2, 1 << (n - 1 - q))
        cs, sn = (f(t / 2).view(B, 1, 1, 1) for f in (torch.cos, torch.sin))
        a, b = w[:, :, :, 0].clone(), w[:, :, :, 1].clone()
        w[:, :, :, 0] = cs * a - sn * b
        w[:, :, :, 1] = sn * a + cs * b

    ladder = torch.ones(1 << n, dtype=torch.float64, device="cuda")
    for i in range(n - 1):
        ladder.view(1 << i, 2, 2, -1)[:, 1, 1].neg_()
    both = torch.zeros(B, 2, 1 << n, dtype=C128, device="cuda")
    psi = torch.zeros(B, 1 << n, dtype=C128, device="cuda")
    psi[:, 0] = 1
    for l in range(L):
        for q in range(n):
            ry(psi, q, th[:, l, q])
        psi *= ladder
    both[:, 0] = psi
    for b in range(B):
        H.add(psi[b], both[b, 1], 1.0)
    energy = (both[:, 0].conj() * both[:, 1]).sum(1).real
    grad = torch.zeros(B, L, n, dtype=torch.float64, device="cuda")
    for l in range(L - 1, -1, -1):
        both *= ladder
        for q in range(n - 1, -1, -1):
            # dE/dt = 2 Re <lambda| dRY(t)/dt RY(t)^-1 |psi>, which is -i Y / 2
            w = both.view(B, 2, 1 << q, 2, 1 << (n - 1 - q))
            grad[:, l, q] = ((w[:, 1, :, 1].conj() * w[:, 0, :, 0]).sum((1, 2)) -
                             (w[:, 1, :, 0].conj() * w[:, 0, :, 1]).sum((1, 2))).real
            ry(both, q, -th[:, l, q])
    return [energy, grad.view(B, -1)]


def exact_adiabatic(c, seed):
    outs = []
    for n, hs in instances(c, seed).items():
        states = []
        for terms in hs:
            e = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
            for coeff, _, zm in terms:
                e += coeff * signs(n, zm)
            psi = torch.full((1 << n,), 2.0 ** (-n / 2), dtype=C128, device="cuda")
            for k in range(c["steps"]):
                s = (k + 0.5) * DT / (1000 * DT)
                half = torch.polar(torch.ones_like(e), -0.5 * DT * s * e)
                psi *= half
                t = -2 * DT * (1 - s)  # H0 = -sum X
                u = np.array([[math.cos(t / 2), -1j * math.sin(t / 2)], [-1j * math.sin(t / 2), math.cos(t / 2)]])
                for q in range(n):
                    apply_matrix(psi, n, (q,), (), u)
                psi *= half
            states.append(psi)
        outs.append(torch.cat(states))
    return outs


def exact_readout(c, seed):
    n = c["n"]
    psi = final_state(n, c["dtype"], seed).to(C128)
    p = psi.real ** 2 + psi.imag ** 2
    energy = 0.0
    for i in range(n - 1):
        m = p.view(1 << i, 2, 2, -1).sum((0, 3))
        energy -= float(m[0, 0] + m[1, 1] - m[0, 1] - m[1, 0])
    for q in range(n):
        v = psi.view(1 << q, 2, -1)
        energy -= 2 * float((v[:, 0].real * v[:, 1].real).sum() + (v[:, 0].imag * v[:, 1].imag).sum())
    group = sorted(int(q) for q in qi.rng(n).permutation(n)[:c["group"]])
    shape, last, keep = [], -1, []
    for q in group:
        shape += [1 << (q - last - 1), 2]
        keep.append(len(shape) - 1)
        last = q
    v = p.view(shape + [1 << (n - 1 - last)])
    v = v.sum([d for d in range(v.dim()) if d not in keep]).reshape(-1)
    norm = float(p.sum())
    return [torch.tensor([energy], dtype=torch.float64), torch.tensor([norm], dtype=torch.float64), v, None]


def exact_density(c, seed):
    n = c["n"]
    dt = np.complex64 if c["dtype"] == "c64" else np.complex128
    psi = torch.from_numpy(qi.random_state(n, seed).astype(dt)).cuda().to(C128)
    rho = (psi[:, None] * psi.conj()[None, :]).reshape(-1)
    noise = sum(np.kron(k, k.conj()) for k in depolarizing())
    for layer in noisy_layers(c):
        for g in layer:
            u = matrix_of(g)
            apply_matrix(rho, 2 * n, g.targets, g.controls, u)
            apply_matrix(rho, 2 * n, [n + q for q in g.targets], [n + q for q in g.controls], u.conj())
        for q in range(n):
            apply_matrix(rho, 2 * n, (q, n + q), (), noise)
    return rho


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("plan", "once"):
        psi = torch.zeros(1 << c["n"], dtype=C128, device="cuda")
        psi[basis_of(c, seed)] = 1
        for g in circuit_of(c, seed):
            apply_matrix(psi, c["n"], g.targets, g.controls, matrix_of(g))
        return psi
    return {"gradient": exact_gradient, "adiabatic": exact_adiabatic, "evolve": exact_evolve,
            "readout": exact_readout, "density": exact_density}[kind](c, seed)
