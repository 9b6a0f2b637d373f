"""The ink rheology's limits: relaxation-time clamps next to 1/2, in FP64, against
the oracle at the FP64 bar, and the iteration's cap."""
import numpy as np
import pytest

import oracle as O

from test_gpu_parity import TOL, assert_close, f32_exact, run_pair

pytestmark = pytest.mark.gpu

SHAPE = (24, 6, 9)


def _sheared(fraction):
    """Ink of the given mass fraction sheared over two decades of amplitude."""
    nx, ny, nz = SHAPE
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    amp = 10.0 ** np.linspace(-3, -1.3, nx)[x]
    u = np.stack([amp * np.sin(2 * np.pi * z / nz), 0.3 * amp * np.cos(2 * np.pi * z / nz), 0 * amp])
    c = np.full((nz, ny, nx), fraction)
    return f32_exact(c, 1.0 - c, u)


def _workload(storage, **rheo):
    return dict(params=dict(velset=1, storage=storage, A=0.01, beta=0.7, tau_amb=0.8), geom=dict(nozzle=0, z_mode=O.Z_PERIODIC),
                rheo=dict(dict(law=O.POWER_LAW, n=0.6, K=0.01, tau_min=0.51, tau_max=2.0), **rheo))


@pytest.mark.parametrize("fraction", [1.0, 0.5, 2.0 ** -36, 0.0])
@pytest.mark.parametrize("above", [2.0 ** -26, 1e-10, 2.0 ** -52])
def test_fp64_viscosity_with_tau_min_next_to_one_half(above, fraction):
    """tau_min - 1/2 below the spacing of FP32 numbers near 1/2."""
    wl = _workload("f64", tau_min=0.5 + above)
    fg, fo, _ = run_pair(SHAPE, wl, 4, "auto", init=_sheared(fraction))
    assert_close(fg, fo, TOL["f64"], label="tau_min 1/2 + %g" % above)


def _capped_nu(nu, r, cap):
    """The viscosity after at most cap steps of Newton's method kept inside the
    bracket, where the converged one is nu (pure power-law ink between its
    clamps): the shear stress over the density follows from nu."""
    law = lambda g: (0.5 + 3 * r["K"] * g ** (r["n"] - 1), 3 * r["K"] * (r["n"] - 1) * g ** (r["n"] - 2))
    g = (nu / r["K"]) ** (1 / (r["n"] - 1))
    s = g * (0.5 + 3 * nu)
    lo, hi = s / r["tau_max"], s / r["tau_min"]
    g = np.clip(np.minimum(2 * s, (s / (3 * r["K"])) ** (1 / r["n"])), lo, hi)
    for _ in range(cap):
        t, dt = law(g)
        dt = np.where((t > r["tau_max"]) | (t < r["tau_min"]), 0.0, dt)
        t = np.clip(t, r["tau_min"], r["tau_max"])
        h = g * t - s
        lo, hi = np.where(h < 0, g, lo), np.where(h < 0, hi, g)
        gn = g - h / (t + g * dt)
        g = np.where((gn > lo) & (gn < hi), gn, 0.5 * (lo + hi))
    return (np.clip(law(g)[0], r["tau_min"], r["tau_max"]) - 0.5) / 3


# nu's own bar in each storage, and room for the FP32 stress noise it carries
@pytest.mark.parametrize("storage,rtol", [("f64", 1e-9), ("f32", 1e-3)])
def test_max_iter_caps_the_iteration(storage, rtol):
    """One step of the iteration instead of sixty, after one time step."""
    wl = _workload(storage, max_iter=1)
    fg, fo, _ = run_pair(SHAPE, wl, 1, "auto", storage=storage, init=_sheared(1.0))
    nu = np.asarray(fo["nu"], dtype=np.float64)
    inside = (0.5 + 3 * nu > 0.52) & (0.5 + 3 * nu < 1.9)
    expect = _capped_nu(nu[inside], wl["rheo"], 1)
    assert np.abs(expect / nu[inside] - 1).max() > 10 * rtol and inside.mean() > 0.5
    assert np.allclose(np.asarray(fg["nu"], dtype=np.float64)[inside], expect, rtol=rtol, atol=0)
