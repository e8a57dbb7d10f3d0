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


# Gaussian widths s of 6.25, 7.5, 10, 12.5, 18 and 22.5 samples: 8 nodes per cell down to 6
@pytest.mark.parametrize("fs,n_s,n_cycles", [(25e6, 803, 5.0), (50e6, 1601, 3.0), (40e6, 1500, 5.0), (50e6, 2001, 5.0),
                                             (40e6, 1502, 9.0), (50e6, 2003, 9.0)])
def test_every_node_count(ur, fs, n_s, n_cycles):
    w = workload(fs, n_s, n_cycles)
    rf, quad, arr, launches = traced(ur, w, 200_000)
    assert np.bincount(arr["el"], minlength=4).min() >= 1024 and launches == 2
    orf, oq = oracle.deposit(w["array"], 1, arr)
    assert rel_l2(rf, orf) <= 4e-6 and rel_l2(quad, oq) <= 4e-6


def test_short_pulses_stay_tap_by_tap(ur):
    """s = 4 samples: no node count interpolates it well enough."""
    w = workload(40e6, 642, 2.0)
    rf, quad, arr, launches = traced(ur, w, 200_000)
    assert np.bincount(arr["el"], minlength=4).min() >= 1024 and launches == 1
    orf, oq = oracle.deposit(w["array"], 1, arr)
    assert rel_l2(rf, orf) <= 4e-6 and rel_l2(quad, oq) <= 4e-6


def test_rows_of_both_kinds_in_one_call(ur):
    """Elements over the scatterers fill their rows, the outer ones receive little.  A row of n arrivals
    deposited tap by tap may add n equal pulses (one scatterer's), n / 2 roundings of the sum on average."""
    w = phantoms.tiny(n_scat=300, with_sphere=False)
    w["scene"]["boundaries"] = []
    sc = w["scene"]["scatterers"]
    sc[10:, 0] = 4e-3 + 0.02 * sc[10:, 0]
    sc[10:, 1] *= 0.2
    sc[:10, :3] = np.column_stack([np.linspace(-4.5e-3, 0.5e-3, 10), np.zeros(10), np.full(10, 0.02)])
    w["array"] = phantoms.array_params(32, 1536, c_bf=1480.0, alpha_m_deg=4.0, alpha_c_deg=4.0)
    rf, quad, arr, launches = traced(ur, w, 3_000_000)
    rows = np.bincount(arr["el"], minlength=32)
    assert launches == 2 and rows.mean() >= 1024
    assert (rows >= 1024).sum() >= 4 and ((rows > 0) & (rows < 1024)).sum() >= 4
    orf, oq = oracle.deposit(w["array"], 1, arr)
    for g, o in ((rf, orf), (quad, oq)):
        for e in np.flatnonzero(rows):
            bar = 4e-6 + (rows[e] / 2 * 2.0 ** -24 if rows[e] < 1024 else 0.0)
            assert rel_l2(g[0, e], o[0, e]) <= bar, (e, rows[e])


def test_batch_through_the_nodes(ur):
    """A batch knows its arrivals on the device only; dense and sparse items in one launch, with a queue
    that holds them and again with the larger queue a longer trace has left behind."""
    import torch
    w = workload(40e6, 1536, 5.0)
    w["angles"] = np.deg2rad(np.array([0.0, 5.0])).astype(np.float32)
    rays = (300_000, 400)
    sim = ur.Simulator(0)
    sim.load(w)
    items = [(0, k, rays[k], k) for k in range(2)]
    want = []
    for k in range(2):
        one = ur.Simulator(0)
        one.load(w)
        _, _, _, rec, _ = one.trace_debug(rays[k], 7, w["max_bounces"], w["max_path"], capacity=4_000_000)
        arr = gpu_records(rec, 4)
        arr = arr[arr["tx"] == k]
        o = oracle.deposit(w["array"], 2, arr)
        want.append((o[0][k], o[1][k], np.bincount(arr["el"], minlength=4)))
    assert want[0][2].min() >= 2048 and want[1][2].max() < 1024
    for _ in range(2):
        sim.batch_plan(items, w["x_px"], w["z_px"], capacity=300_000)
        rf, quad = sim.batch_trace(7, w["max_bounces"], w["max_path"])
        n, _ = sim.batch_status()
        assert n == want[0][2].sum() + want[1][2].sum()
        for k in range(2):
            assert rel_l2(rf[k].double().cpu().numpy(), want[k][0]) <= 4e-6
            assert rel_l2(quad[k].double().cpu().numpy(), want[k][1]) <= 4e-6
        sim.trace(2_000_000, 1, w["max_bounces"], w["max_path"])


@pytest.mark.parametrize("fs,n_cycles", [(50e6, 5.0), (40e6, 5.0), (50e6, 3.0), (25e6, 5.0), (50e6, 9.0)])
def test_weak_ends_of_the_pulse(ur, fs, n_cycles):
    """A plane's echo at one time, every sample relative to its own envelope (4e-6 of the peak at the cut):
    no further off than one tap evaluated in FP32, where the carrier's argument (h half-cycles at the cut,
    two rounded factors and their product) and the Gaussian's (12.5, three roundings) are rounded."""
    worst = 0.0
    for depth in 0.0101 + 13.7e-6 * np.arange(12):   # times all over a cell
        w = phantoms.single_plane(depth=depth, lower=phantoms.BONE, n_el=4, n_s=1024, pitch=1e-3, fs=fs, n_cycles=n_cycles)
        rf, quad, arr, launches = traced(ur, w, 40_000)
        t = np.unique(arr["t"])
        assert launches == 2 and t.size == 1 and np.bincount(arr["el"], minlength=4).min() >= 1024
        s = n_cycles / (4 * w["array"]["f0"]) * fs
        n = np.arange(1024)
        n = n[np.abs(n - t[0]) <= 5 * s]
        u = n - t[0]
        env, phase = np.exp(-u * u / (2 * s * s)), 2 * np.pi * w["array"]["f0"] / fs * u
        carrier = np.sin(phase) - 1j * np.cos(phase)
        for e in range(4):
            g = (rf[0, e] + 1j * quad[0, e])[n] / env
            mid = np.abs(u) < s
            amp = np.vdot(carrier[mid], g[mid]) / mid.sum()   # the row's amplitude
            worst = max(worst, np.abs(g / amp - carrier).max())
    h = 5 * s * 2 * w["array"]["f0"] / fs
    assert worst <= (1.5 * np.pi * h + 3 * 12.5 + 8) * 2.0 ** -24


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
