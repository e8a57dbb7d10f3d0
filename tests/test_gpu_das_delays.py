"""The delay-and-sum's interpolation weights, its independence of the other images of a batch, and
arrays of the largest element count."""
import numpy as np
import pytest

import oracle
import phantoms
from _parity import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ur():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as u
    return u


@pytest.mark.parametrize("n_el", [3072, 3073, 4096])
def test_convex_arrays_of_many_elements(ur, n_el):
    """Every array that set_array takes can be beamformed.  Bar as in the tiles' tests."""
    import torch
    A = phantoms.array_params(n_el, 64, pitch=1e-5)
    A["radius"] = 0.05
    rng = np.random.default_rng(n_el)
    rf, quad = (rng.standard_normal((1, n_el, 64)).astype(np.float32) for _ in range(2))
    x = np.linspace(-2e-3, 2e-3, 19).astype(np.float32)
    z = np.linspace(1e-4, 1.2e-3, 7).astype(np.float32)
    tx = [(ur.TX_DIVERGING, 0.0, -0.04)]
    sim = ur.Simulator(0)
    sim.set_array(A)
    sim.set_transmits(tx)
    g = sim.beamform(torch.from_numpy(rf).cuda(), torch.from_numpy(quad).cuda(), x, z)[0].double().cpu().numpy()
    o = oracle.beamform(A, np.zeros(1, np.float32), rf.astype(np.float64), quad.astype(np.float64), x, z, transmits=tx)
    assert np.abs(o).max() > 0
    assert rel_l2(g[..., 0] + 1j * g[..., 1], o) <= 4 * (3 + np.sqrt(n_el)) * 2.0 ** -24
