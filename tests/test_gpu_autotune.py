"""The autotuner starts from what an untuned trace runs with, so its choice is not slower (5 % for the
clock; each side the best of several traces, taken in turn)."""
import numpy as np
import pytest

import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["smooth", "rough"])
def test_tuned_trace_is_not_slower_than_untuned(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as ur
    w = phantoms.layered(n_scat=20_000)
    if kind == "rough":
        w["scene"]["media"][3, 3] = 0.5
    plain, tuned = ur.Simulator(0), ur.Simulator(0)
    for sim in (plain, tuned):
        sim.load(w)
    best = tuned.autotune(1_000_000)
    assert best["cell_xy"] > 0 and best["cell_y"] > 0 and best["cell_z"] > 0 and 1 <= best["resolve_batch"] <= 32
    ms = [[], []]
    out = [sim.trace(1_000_000, 0, 8, stats=True) for sim in (plain, tuned)]
    assert out[0][2] == out[1][2]
    for _ in range(7):
        for sim, t in zip((plain, tuned), ms):
            sim.set_profiling(True)
            sim.trace(1_000_000, 0, 8)
            t.append(sim.profile()["trace"][0])
    assert min(ms[1]) <= 1.05 * min(ms[0])
