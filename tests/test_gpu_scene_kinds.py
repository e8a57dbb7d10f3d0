"""One tracer instantiation against another on the same scenes: a batch of a smooth, a rough and a meshed
scene (traced together by the extended mesh tracer) against each alone, and convex arrays on thin,
wide and lopsided grids against one cell.  Counters are equal; channel data are the same arrivals summed
in another order: a few ulp of the row's largest sample."""
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


def test_batch_of_scenes_of_other_kinds(ur):
    import torch
    A = phantoms.array_params(128, 4096, fs=50e6)
    ws = [phantoms.layered(seed=1, n_scat=2500), phantoms.layered(seed=2, n_scat=2000), phantoms.paper_mesh_like(n_scat=2000, subdiv=2, n_seg=16)]
    ws[1]["scene"]["media"][3, 3] = 0.5
    angles = np.deg2rad(np.array([0.0, -9.0])).astype(np.float32)
    for w in ws:
        w.update(array=A, angles=angles)
    sim = ur.Simulator(0)
    for k, w in enumerate(ws):
        sim.load(w, slot=k)
    sim.batch_plan([(k, t, 9001, t) for k in range(3) for t in range(2)], ws[0]["x_px"], ws[0]["z_px"], capacity=200_000)
    rf, quad = sim.batch_trace(5, 8)
    _, st = sim.batch_status()
    total = {}
    for k, w in enumerate(ws):
        one = ur.Simulator(0)
        one.load(w)
        r, q, s = one.trace(9001, 5, 8, stats=True)
        assert s["arrivals"] > 0
        for a, b in ((rf, r), (quad, q)):
            assert torch.allclose(a[2 * k:2 * k + 2], b, rtol=0, atol=1e-5 * float(b.abs().max())), k
        total = {f: total.get(f, 0) + v for f, v in s.items()}
    assert st == total


@pytest.mark.parametrize("kind", ["diverging", "synthetic"])
def test_convex_array_on_every_grid(ur, kind):
    w = phantoms.paper_like(n_scat=3000, convex=True)
    w["transmits"] = [(ur.TX_DIVERGING, 2e-3, -0.05)] if kind == "diverging" else [(ur.TX_SYNTHETIC, float(e), 0.0) for e in (3, 64)]
    out = []
    for tuning in (dict(cell_xy=1.0, cell_y=1.0, cell_z=1.0), {}, dict(cell_xy=0.5 * R_S, cell_y=9 * R_S, cell_z=3 * R_S),
                   dict(cell_xy=11 * R_S, cell_y=0.4 * R_S, cell_z=50 * R_S), dict(cell_xy=37 * R_S, cell_y=41 * R_S, cell_z=2 * R_S)):
        sim = ur.Simulator(0)
        sim.set_tuning(**tuning)
        sim.load(w)
        _, _, st, rec, ph = sim.trace_debug(20_001, 5, w["max_bounces"], w["max_path"])
        rec = np.stack([rec[k].cpu().numpy().view(np.uint32) for k in ("row", "ray", "event", "t_hi", "t_lo", "amp")], 1)
        out.append((st, rec[np.lexsort(rec.T[::-1])], ph.cpu().numpy()))
    assert out[0][0]["candidates"] > 100
    for st, rec, ph in out[1:]:
        assert st == out[0][0] and np.array_equal(rec, out[0][1]) and np.array_equal(ph, out[0][2])
