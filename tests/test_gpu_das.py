"""Delay-and-sum at the edges of its tiles: narrow, odd and large images, every chunk of transmits,
small element counts, the ends of the recording, and pixels outside the fixed-point delays' range.

Tolerance: white-noise channel data, N = transmits x elements terms per pixel in FP32.  An
interpolation weight carries at most 2 x 2^-24 (the receive delay's fraction and the weight
itself, each rounded to 24 bits) times a sample difference (1.4 RMS); a running sum adds 2^-24
of its partial value per term, which for random terms is at most sqrt(N) of a term's share of
the result.  The bar is 4 (3 + sqrt(N)) 2^-24."""
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


def image(ur, A, tx, rf, quad, x, z):
    import torch
    sim = ur.Simulator(0)
    sim.set_array(A)
    sim.set_transmits(tx)
    iq, env, db = sim.beamform(torch.from_numpy(rf).cuda(), torch.from_numpy(quad).cuda(), x, z, 60.0)
    g = iq.double().cpu().numpy()
    g = g[..., 0] + 1j * g[..., 1]
    assert np.allclose(env.double().cpu().numpy(), np.abs(g), rtol=1e-6, atol=0, equal_nan=True)
    return g, db.cpu().numpy()


CASES = [  # n_el, n_s, n_tx, nx, nz, radius
    (33, 16, 1, 1, 700, 0.0),       # shortest recording, one column: lanes along depth
    (1, 200, 2, 3, 45, 0.0),        # one element
    (17, 800, 3, 33, 9, 0.0),       # one pixel past a warp
    (128, 3200, 4, 31, 33, 0.0),
    (64, 1536, 5, 100, 7, 0.05),
    (97, 2999, 6, 65, 17, 0.0),
    (48, 1000, 7, 40, 40, 0.0),
    (130, 1111, 9, 37, 21, 0.05),
    (40, 900, 17, 16, 50, 0.0),
    (20, 640, 1, 700, 500, 0.0),    # large image: one warp per pixel group
    (128, 8192, 1, 24, 24, 0.0),
]


@pytest.mark.parametrize("n_el,n_s,n_tx,nx,nz,radius", CASES)
def test_das_tiles(ur, n_el, n_s, n_tx, nx, nz, radius):
    A = phantoms.array_params(n_el, n_s)
    if radius:
        A["radius"] = radius
    rng = np.random.default_rng(n_el * 1000 + n_tx)
    rf = rng.standard_normal((n_tx, n_el, n_s)).astype(np.float32)
    quad = rng.standard_normal((n_tx, n_el, n_s)).astype(np.float32)
    kinds = [(ur.TX_PLANE, 0.02, 0.0), (ur.TX_DIVERGING, 1e-3, -8e-3), (ur.TX_FOCUSED, -2e-3, 12e-3),
             (ur.TX_SYNTHETIC, float(n_el // 2), 0.0), (ur.TX_PLANE, -0.1, 0.0), (ur.TX_DIVERGING, 0.0, -1e3)]
    tx = [kinds[k % len(kinds)] for k in range(n_tx)]
    half = 0.6 * n_el * A["pitch"]
    x = np.linspace(-half, 0.9 * half, nx).astype(np.float32) if nx > 1 else np.zeros(1, np.float32)
    z = np.linspace(1e-4, 1.1 * A["c_bf"] * n_s / (2 * A["fs"]), nz).astype(np.float32)   # past the last sample
    g, _ = image(ur, A, tx, rf, quad, x, z)
    angles = np.array([a if k == ur.TX_PLANE else 0.0 for k, a, _ in tx], np.float32)
    o = oracle.beamform(A, angles, rf.astype(np.float64), quad.astype(np.float64), x, z,
                        transmits=tx)
    assert np.abs(o).max() > 0
    assert rel_l2(g, o) <= 4 * (3 + np.sqrt(n_tx * n_el)) * 2.0 ** -24


def test_das_recording_ends(ur):
    """One element over its own column with delays that are whole samples: sample 0 and the last
    one count in full, anything past it not at all."""
    n_s = 100
    A = phantoms.array_params(1, n_s, f0=65536.0, fs=524288.0, c_bf=1024.0, pitch=1e-3)
    z = (np.array([0.0, 1.0, 1.5, n_s - 2, n_s - 1, n_s - 1 + 1 / 64, n_s]) / 1024).astype(np.float32)
    rf = (1.0 + np.arange(n_s, dtype=np.float32)).reshape(1, 1, n_s)
    g, _ = image(ur, A, [(ur.TX_PLANE, 0.0, 0.0)], rf, -rf, np.zeros(1, np.float32), z)
    want = np.array([1, 2, 2.5, n_s - 1, n_s, 0, 0])
    assert np.array_equal(g[:, 0], want - 1j * want)


def test_das_pixels_out_of_range(ur):
    """Pixels kilometres away or not finite leave the other pixels alone."""
    A = phantoms.array_params(32, 500)
    rng = np.random.default_rng(3)
    rf, quad = (rng.standard_normal((2, 32, 500)).astype(np.float32) for _ in range(2))
    x = np.linspace(-4e-3, 4e-3, 9).astype(np.float32)
    z = np.linspace(1e-3, 8e-3, 5).astype(np.float32)
    tx = [(ur.TX_PLANE, 0.1, 0.0), (ur.TX_DIVERGING, 0.0, -1e-2)]
    ref, _ = image(ur, A, tx, rf, quad, x, z)
    xs = x.copy()
    xs[[0, 4, 6]] = 5e3, np.nan, -3e9
    g, _ = image(ur, A, tx, rf, quad, xs, z)
    keep = [1, 2, 3, 5, 7, 8]
    assert np.array_equal(g[:, keep], ref[:, keep])
    assert np.all(g[:, [0, 6]] == 0) and np.all(np.isnan(g[:, 4]))
