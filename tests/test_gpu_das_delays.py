"""The delay-and-sum's interpolation weights, its independence of the other images of a batch, and
arrays of the largest element count."""
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


@pytest.mark.parametrize("kind", ["plane", "diverging", "focused"])
def test_weight_is_rounded_once(ur, kind):
    """One element, samples 0 1 0 1 ...: where the delay's sample is even, the pixel's value is the
    interpolation weight itself.  A weight in [0, 1) rounded once to FP32 is off by at most 2^-25;
    the delays' own errors (32.32 fixed point, square roots) have to stay far below: 2^-28 in all."""
    import torch
    n_s = 8192
    A = phantoms.array_params(1, n_s)
    tx = {"plane": (ur.TX_PLANE, 0.2, 0.0), "diverging": (ur.TX_DIVERGING, 1e-3, -8e-3),
          "focused": (ur.TX_FOCUSED, 2e-3, 0.3)}[kind]
    x = np.linspace(-15e-3, 16e-3, 701).astype(np.float32)
    z = np.linspace(2e-3, 0.14, 499).astype(np.float32)
    rf = torch.zeros(1, 1, n_s, device="cuda")
    rf[..., 1::2] = 1.0
    sim = ur.Simulator(0)
    sim.set_array(A)
    sim.set_transmits([tx])
    v = sim.beamform(rf, torch.zeros_like(rf), x, z)[0][..., 0].double().cpu().numpy()
    q = A["fs"] / A["c_bf"]
    X, Z = x.astype(np.float64)[None, :], z.astype(np.float64)[:, None]
    R = np.sqrt(X * X + Z * Z)   # the element's centre is the origin
    if kind == "plane":
        a = float(np.float32(tx[1]))
        T = X * np.sin(a) + Z * np.cos(a)
    else:
        vx, vz = float(np.float32(tx[1])), float(np.float32(tx[2]))
        r, re = np.sqrt((X - vx) ** 2 + (Z - vz) ** 2), np.hypot(vx, vz)
        T = r - re if kind == "diverging" else re + np.where(Z >= vz, r, -r)
    tau = (T + R) * q
    i0 = np.floor(tau)
    even = (i0 % 2 == 0) & (tau > 0) & (tau < n_s - 1)
    assert even.sum() > 100_000
    assert np.abs(v - (tau - i0))[even].max() <= 2.0 ** -25 + 2.0 ** -28


def test_columns_far_apart_and_past_a_warp(ur):
    """33 columns over 0.2 m cost no more each than 12 do: neither the lanes of a second warp without
    pixels nor gathers without a shared cache line (1.4 times as much with warps of 32 columns)."""
    import torch
    A = phantoms.array_params(64, 8192)
    sim = ur.Simulator(0)
    sim.set_array(A)
    sim.set_plane_waves(np.deg2rad(np.linspace(-10, 10, 31)).astype(np.float32))
    rf, quad = (torch.randn(31, 64, 8192, device="cuda") for _ in range(2))
    z = torch.linspace(1e-3, 0.15, 2000, device="cuda")

    def time(nx):
        x = torch.linspace(-0.1, 0.1, nx, device="cuda")
        out = [torch.empty(2000, nx, 2, device="cuda")] + [torch.empty(2000, nx, device="cuda") for _ in range(2)]
        t = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            sim.beamform(rf, quad, x, z, 60.0, *out)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    assert time(33) / 33 <= 1.15 * time(12) / 12


@pytest.mark.parametrize("n_el", [3072, 3073, 4096])
def test_convex_arrays_of_many_elements(ur, n_el):
    """Every array that set_array takes can be beamformed.  Bar as in the tiles' tests."""
    import torch
    A = phantoms.array_params(n_el, 64, pitch=1e-5)
    A["radius"] = 0.05
    rng = np.random.default_rng(n_el)
    rf, quad = (rng.standard_normal((1, n_el, 64)).astype(np.float32) for _ in range(2))
    x = np.linspace(-2e-3, 2e-3, 19).astype(np.float32)
    z = np.linspace(1e-4, 1.2e-3, 7).astype(np.float32)
    tx = [(ur.TX_DIVERGING, 0.0, -0.04)]
    sim = ur.Simulator(0)
    sim.set_array(A)
    sim.set_transmits(tx)
    g = sim.beamform(torch.from_numpy(rf).cuda(), torch.from_numpy(quad).cuda(), x, z)[0].double().cpu().numpy()
    o = oracle.beamform(A, np.zeros(1, np.float32), rf.astype(np.float64), quad.astype(np.float64), x, z, transmits=tx)
    assert np.abs(o).max() > 0
    assert rel_l2(g[..., 0] + 1j * g[..., 1], o) <= 4 * (3 + np.sqrt(n_el)) * 2.0 ** -24
