"""Deposit through interpolation nodes: which rows take it, every node count, weak ends of the pulse,
amplitudes that are not finite, batches, and several simulators at once.

Tolerance against the oracle's FP64 deposit of the GPU's own records, as for the other deposits: a
work item adds up to 4096 arrivals in FP32, sqrt(4096) 2^-24 = 4e-6 relative if they share a cell."""
import threading

import numpy as np
import pytest

import oracle
import phantoms
from _parity import gpu_records, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ur():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_05828_gb300 as u
    return u


def workload(fs, n_s, n_cycles, n_scat=400):
    w = phantoms.tiny(n_scat=n_scat)
    w["array"] = phantoms.array_params(4, n_s, fs=fs, n_cycles=n_cycles, c_bf=1480.0, alpha_m_deg=60.0, alpha_c_deg=60.0,
                                       pitch=1e-3)
    return w


def traced(ur, w, n_rays, seed=3):
    sim = ur.Simulator(0)
    sim.load(w)
    sim.set_profiling(True)
    rf, quad, st, rec, _ = sim.trace_debug(n_rays, seed, w["max_bounces"], w["max_path"], capacity=4_000_000)
    launches = sim.profile()["deposit"][1]   # 2: the node kernel ran as well
    return rf.double().cpu().numpy(), quad.double().cpu().numpy(), gpu_records(rec, w["array"]["n_el"]), launches


def test_amplitudes_that_are_not_finite_keep_to_their_taps(ur):
    """A scatterer whose amplitude is NaN or infinite spoils the samples its pulses cover, no others."""
    w = workload(40e6, 1536, 5.0)
    w["scene"]["scatterers"][7, 3] = np.nan
    w["scene"]["scatterers"][11, 3] = np.inf
    rf, quad, arr, launches = traced(ur, w, 200_000)
    assert launches == 2 and np.bincount(arr["el"], minlength=4).min() >= 1024
    bad = ~np.isfinite(arr["amp"])
    assert 0 < bad.sum() < arr.size
    K = 5.0 * 5.0 / (4 * w["array"]["f0"]) * w["array"]["fs"]
    hit = np.zeros((4, 1536), bool)
    for a in arr[bad]:
        hit[a["el"], max(0, int(np.ceil(a["t"] - K))):int(np.floor(a["t"] + K)) + 1] = True
    assert hit.any() and not hit.all()
    orf, oq = oracle.deposit(w["array"], 1, arr[~bad])
    for g, o in ((rf, orf), (quad, oq)):
        assert np.array_equal(np.isfinite(g[0]), ~hit)
        assert rel_l2(g[0][~hit], o[0][~hit]) <= 4e-6


def test_simulators_of_other_row_lengths_in_other_threads(ur):
    """The node kernel's shared memory differs with the row's length; calls of several threads do not
    take one another's."""
    import torch
    errors = []

    def work(n_s):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                sim = ur.Simulator(0, stream=stream)
                sim.load(workload(40e6, n_s, 5.0))
                rf, quad = sim.trace(60_000, 3, 4)
                for k in range(400):
                    sim.trace(60_000, 3, 4, rf=rf, quad=quad)
                sim.sync()
        except Exception as e:   # noqa: BLE001 - reported below
            errors.append(e)

    ts = [threading.Thread(target=work, args=(n,)) for n in (2300, 8192, 3000, 6000)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
