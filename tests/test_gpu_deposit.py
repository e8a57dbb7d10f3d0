"""The pulse deposit through interpolation nodes (rows of many arrivals) against the oracle's FP64
deposit of the GPU's own arrival records: pulses of whole and fractional half-widths, rows whose
length is no multiple of a cell, arrivals at both ends of the row, and echoes that share one time.

Tolerance: the Gaussian's interpolation error is below 2e-8 of the peak; a cell adds up to 4096
arrivals of one work item in FP32, sqrt(4096) 2^-24 = 4e-6 relative if they all share a cell."""
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


@pytest.mark.parametrize("fs,n_s,n_cycles,n_scat", [(40e6, 1536, 5.0, 400), (50e6, 1001, 5.0, 400), (40e6, 642, 2.0, 400),
                                                    (25e6, 803, 9.0, 400), (40e6, 1536, 5.0, 0), (40e6, 90, 5.0, 400)])
def test_node_deposit_matches_oracle(ur, fs, n_s, n_cycles, n_scat):
    w = phantoms.tiny(n_scat=max(n_scat, 1))
    if not n_scat:
        w["scene"]["scatterers"] = np.zeros((0, 4), np.float32)   # planar and spherical echoes only
    if n_s < 100:
        w["scene"]["scatterers"][:, 2] = 1e-3 + 1e-3 * np.arange(n_scat) / n_scat   # echoes inside a short row
    w["array"] = phantoms.array_params(4, n_s, fs=fs, n_cycles=n_cycles, c_bf=1480.0, alpha_m_deg=60.0, alpha_c_deg=60.0,
                                       pitch=1e-3)
    n = 200_000 if n_scat else 1_000_000
    sim = ur.Simulator(0)
    sim.load(w)
    rf, quad, st, rec, _ = sim.trace_debug(n, 3, w["max_bounces"], w["max_path"], capacity=4_000_000)
    arr = gpu_records(rec, 4)
    assert np.bincount(arr["el"], minlength=4).min() >= 1024      # every row goes through the nodes
    orf, oq = oracle.deposit(w["array"], 1, arr)
    assert rel_l2(rf.double().cpu().numpy(), orf) <= 4e-6
    assert rel_l2(quad.double().cpu().numpy(), oq) <= 4e-6
