"""The ink rheology's limits: relaxation-time clamps next to 1/2, in FP64, against
the oracle at the FP64 bar."""
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
