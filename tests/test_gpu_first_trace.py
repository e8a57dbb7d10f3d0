"""The first trace after set_array costs what one after new transmits costs: the deposit's node plan
is made only for a call that uses it, and is quick.  (A plan that evaluates every Gaussian afresh
took a quarter of a millisecond of host time.)"""
import time

import numpy as np
import pytest

import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fs,n_rays,dense", [(40e6, 2_000, False), (40e6, 400_000, True), (50e6, 400_000, True)])
def test_first_trace_of_an_array(fs, n_rays, dense):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as ur
    w = phantoms.tiny(n_scat=400)
    w["array"] = phantoms.array_params(4, 1536, fs=fs, c_bf=1480.0, pitch=1e-3, alpha_m_deg=60.0, alpha_c_deg=60.0)
    sim = ur.Simulator(0)
    sim.load(w)
    rf, quad, st = sim.trace(n_rays, 0, 4, stats=True)
    assert (st["arrivals"] >= 4 * 1024) == dense

    def first(new_array):
        if new_array:
            sim.set_array(w["array"])
        sim.set_plane_waves(w["angles"])   # either way the transmit tables are made again
        torch.cuda.synchronize()
        t = time.perf_counter()
        sim.trace(n_rays, 0, 4, rf=rf, quad=quad)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    for new in (True, False):
        first(new)
    t = np.array([[first(True), first(False)] for _ in range(25)])
    assert np.median(t[:, 0] - t[:, 1]) < 0.1e-3
