"""Default scatterer-grid cells where the scatterers do not fill their bounding box: a dense lesion
with one scatterer far outside the field, speckle in two places.  The trace with the defaults takes
at most half as long again as with columns of 6 capture radii (24 times as long in the first scene by
the box's density alone), and finds the same events."""
import numpy as np
import pytest

import phantoms

pytestmark = pytest.mark.gpu

R_S = 1e-4


@pytest.fixture(scope="module")
def ur():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as u
    return u


def cloud(name):
    rng, box = np.random.default_rng(3), phantoms.uniform_scatterers
    if name == "far":
        return np.concatenate([box(rng, 50_000, ((-4e-3, 4e-3), (-2.5e-3, 2.5e-3), (16e-3, 24e-3))),
                               np.array([[0.3, 0.2, 59e-3, 0.5]], np.float32)])
    return np.concatenate([box(rng, 25_000, ((x - 2e-3, x + 2e-3), (-2.5e-3, 2.5e-3), (z - 2e-3, z + 2e-3)))
                           for x, z in ((-10e-3, 20e-3), (12e-3, 50e-3))])


@pytest.mark.parametrize("name", ["far", "two"])
@pytest.mark.parametrize("kind", ["smooth", "rough", "bone"])
def test_default_cells_of_clustered_scatterers(ur, kind, name):
    w = phantoms.paper_like(n_scat=10) if kind == "bone" else phantoms.layered(n_scat=10)
    if kind == "rough":
        w["scene"]["media"][3, 3] = 0.5
    w["scene"]["scatterers"] = cloud(name)
    w["angles"] = np.deg2rad(np.array([10.0])).astype(np.float32)
    ms, stats = [], []
    y = {"smooth": 0.3, "rough": 2.0, "bone": 6.0}[kind]
    for tuning in ({}, dict(cell_xy=6 * R_S, cell_y=y * R_S, cell_z=4 * R_S)):
        sim = ur.Simulator(0)
        sim.set_tuning(**tuning)
        sim.load(w)
        rf, quad, st = sim.trace(500_000, 1, w["max_bounces"], w["max_path"], stats=True)
        t = []
        for _ in range(5):
            sim.set_profiling(True)
            sim.trace(500_000, 1, w["max_bounces"], w["max_path"], rf=rf, quad=quad)
            t.append(sim.profile()["trace"][0])
        ms.append(min(t))
        stats.append(st)
    assert stats[0] == stats[1] and stats[0]["candidates"] > 100_000
    assert ms[0] <= 1.5 * ms[1], ms
