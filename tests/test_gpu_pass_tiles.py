"""Specialised pass kernels whose CTAs take several tiles each (2048 tiles, or
1500 members of one tile; 2 CTAs per SM are resident), so that a tile's last
transpose meets the next tile's first: against the generic kernels on the same
device, whose transposes all meet, within 4 u per gate of the largest amplitude
(u = 2^-24, double-float 2^-46), and equal from run to run."""
import pytest

from paper_2009_01845_gb300 import inputs as qi
from test_gpu_passes import diagonals, low_two_qubit

pytestmark = pytest.mark.gpu

UNIT = {"c128": 2.0 ** -46, "c64": 2.0 ** -24}


def layers(n, r, long):
    return qi.random_layer_circuit(n, 6 if long else 3, seed=int(r.integers(100)))


@pytest.fixture(scope="module")
def qs():
    from paper_2009_01845_gb300 import qsim
    qsim.load(build_if_missing=True)
    yield qsim
    qsim.jit_set_policy("tiered")


@pytest.mark.parametrize("dtype,n,batch", [("c64", 24, 1), ("c64", 13, 1500), ("c128", 23, 1), ("c128", 12, 1500)])
@pytest.mark.parametrize("circuit", [low_two_qubit, diagonals, layers])
def test_tile_after_tile(qs, circuit, dtype, n, batch):
    import torch
    gates = circuit(n, qi.rng(5 * n), dtype == "c64")
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn(batch << n, dtype=torch.complex64 if dtype == "c64" else torch.complex128, device="cuda",
                      generator=g)
    runs = []
    for policy in ("off", "sync", "sync", "sync"):
        qs.jit_set_policy(policy)
        before = qs.jit_stats()
        st = qs.State(n, batch=batch, dtype=dtype, tensor=psi.clone()).apply(gates, mode="tiled")
        torch.cuda.synchronize()
        after = qs.jit_stats()
        assert after["failed"] == before["failed"]
        if policy == "sync":
            assert after["generic_launches"] == before["generic_launches"]
            assert after["specialised_launches"] > before["specialised_launches"]
        runs.append(st.tensor)
    off, first = runs[:2]
    assert float((first - off).abs().max()) <= 4 * UNIT[dtype] * len(gates) * float(off.abs().max())
    for again in runs[2:]:
        assert torch.equal(again, first)
