"""The tracer's column walk finds the same scatterer events whatever the grid: counters and
per-arrival records with the default cells, thin, wide and lopsided ones against one single cell
(every scatterer tested against every segment inside the scatterers' box), on scenes whose rays
stay in the xz plane, leave it, or travel mostly along y, and in a batch of several scenes.
Everything compared is a count or a record of the same arithmetic: equality, no tolerance."""
import numpy as np
import pytest

import phantoms

pytestmark = pytest.mark.gpu

R_S = 1e-4
ONE_CELL = dict(cell_xy=1.0, cell_y=1.0, cell_z=1.0)
GRIDS = {"default": {}, "thin_x": dict(cell_xy=0.5 * R_S, cell_y=9 * R_S, cell_z=3 * R_S),
         "thin_y": dict(cell_xy=11 * R_S, cell_y=0.4 * R_S, cell_z=50 * R_S),
         "wide": dict(cell_xy=37 * R_S, cell_y=41 * R_S, cell_z=2 * R_S)}


@pytest.fixture(scope="module")
def ur():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as u
    return u


def scene(name):
    if name == "smooth":
        return phantoms.layered(n_scat=3000, n_rays=6001, angles_deg=(0.0, 9.0, -24.0))
    if name == "rough":
        w = phantoms.layered(n_scat=3000, n_rays=6001, angles_deg=(4.0, -24.0))
        w["scene"]["media"][1:, 3] = 0.5
        return w
    if name == "sphere":
        w = phantoms.paper_like(n_scat=3000, n_rays=6001)
        w["angles"] = w["angles"][::8].copy()
        return w
    if name == "along_y":   # one wide column of scatterers: rays scattered by the bone cross it mostly along y
        w = phantoms.tiny(n_scat=4000, n_rays=20_001)
        w["scene"]["scatterers"][:, 0] *= 0.05
        w["scene"]["scatterers"][:, 1] *= 8.0
        w["scene"]["media"][2, 3] = 1.5
        return w
    return phantoms.paper_mesh_like(n_scat=2000, n_rays=2001, subdiv=2, n_seg=16)


def run(ur, w, tuning):
    sim = ur.Simulator(0)
    sim.set_tuning(**tuning)
    sim.load(w)
    _, _, st, rec, ph = sim.trace_debug(w["n_rays"], 5, w["max_bounces"], w["max_path"])
    rec = np.stack([rec[k].cpu().numpy().view(np.uint32) for k in ("row", "ray", "event", "t_hi", "t_lo", "amp")], 1)
    return st, rec[np.lexsort(rec.T[::-1])], ph.cpu().numpy()


@pytest.mark.parametrize("name", ["smooth", "rough", "sphere", "along_y", "mesh"])
def test_every_grid_finds_the_same_events(ur, name):
    w = scene(name)
    st, rec, ph = run(ur, w, ONE_CELL)
    assert st["candidates"] > 100 and st["arrivals"] > 0
    for g, tuning in GRIDS.items():
        st2, rec2, ph2 = run(ur, w, tuning)
        assert st2 == st, g
        assert np.array_equal(rec2, rec) and np.array_equal(ph2, ph), g


def test_batch_of_scenes_matches_single_scene_launches(ur):
    """Scenes read per lane (a batch of several) and as kernel constants (one scene) trace alike."""
    import torch
    ws = [phantoms.layered(seed=k, n_scat=2000 + 500 * k, angles_deg=(0.0, 7.0), bone_r=(4 + k) * 1e-3) for k in range(2)]
    sim = ur.Simulator(0)
    for k, w in enumerate(ws):
        sim.load(w, slot=k)
    items = [(k, t, 7001, t) for k in range(2) for t in range(2)]
    sim.batch_plan(items, ws[0]["x_px"], ws[0]["z_px"], capacity=200_000)
    rf, quad = sim.batch_trace(5, 8)
    _, st = sim.batch_status()
    tot = {}
    for k, w in enumerate(ws):
        one = ur.Simulator(0)
        one.load(w)
        r1, q1, s1 = one.trace(7001, 5, 8, stats=True)
        for a, b in ((rf, r1), (quad, q1)):   # summed in another order: a few ulp of the row's largest sample
            assert torch.allclose(a[2 * k:2 * k + 2], b, rtol=0, atol=1e-5 * float(b.abs().max()))
        tot = {f: tot.get(f, 0) + v for f, v in s1.items()}
    assert st == tot


def test_debug_trace_without_path_hashes(ur):
    """path_hash is nullable: the records are the same without it."""
    w = scene("smooth")
    sim = ur.Simulator(0)
    sim.load(w)
    _, _, st, rec, ph = sim.trace_debug(2000, 5, w["max_bounces"], w["max_path"])
    _, _, st2, rec2, none = sim.trace_debug(2000, 5, w["max_bounces"], w["max_path"], path_hash=False)
    key = lambda r: np.sort(r["ray"].cpu().numpy().astype(np.int64) << 32 | r["event"].cpu().numpy().view(np.uint32))
    assert none is None and st2 == st and np.array_equal(key(rec2), key(rec))
