"""Segments that end on a column's side: a column visit accepts no closest approach past the
segment's end, however slowly the ray crosses the columns.

Plane waves tilted by 1e-5 to 1e-3 rad meet a plane inside a dense sheet of scatterers.  Where
a ray's end point rounds into the next column, the side's distance along the ray is wrong by
ulp(x) / sin(angle), up to a capture radius; narrow columns make that common (about one ray in
10^4).  Against columns wider than the scene (no side on the way) every count is the same."""
import numpy as np
import pytest

import phantoms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ur():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as u
    return u


@pytest.mark.parametrize("rough", [0.0, 0.3])
@pytest.mark.parametrize("angle", [1e-5, -1e-4, 1e-3])
def test_no_event_past_the_end_of_a_segment(ur, angle, rough):
    rng = np.random.default_rng(1)
    w = phantoms.single_plane(depth=0.02, n_el=128, n_s=3200)
    w["scene"]["media"][1, 3] = rough   # the extended tracer
    sc = phantoms.uniform_scatterers(rng, 200_000, ((-19e-3, 19e-3), (-2e-3, 2e-3), (19.95e-3, 20.1e-3)))
    w["scene"]["scatterers"] = sc
    w["angles"] = np.array([angle], np.float32)
    stats = []
    for cell in (1.0, 1e-5):
        sim = ur.Simulator(0)
        sim.set_tuning(cell_xy=cell, cell_y=2e-4, cell_z=1.0)
        sim.load(w)
        stats.append(sim.trace(1_000_000, 3, 0, stats=True)[2])
    assert stats[0]["candidates"] > 1_000_000
    assert stats[1] == stats[0]
