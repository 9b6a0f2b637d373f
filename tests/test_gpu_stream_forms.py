"""The phase-by-phase path's stream kernels on both sides of each size where its
form changes (four threads to a site, one thread with the nozzle's and the top's
rules, one thread without them, the top plane apart), against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2102_02655_gb300 import inputs as I

from test_gpu_parity import FIELDS, TOL, assert_close, f32_exact, run_pair
from test_gpu_storage16 import HYDRO, TOL16

pytestmark = pytest.mark.gpu

BARS = {"f64": (TOL["f64"], FIELDS), "f32": (TOL["f32"], tuple(k for k in FIELDS if k != "nu")), "f16dev": (TOL16, HYDRO)}
# the last size of one form and the first of the next: 19,456, 77,824, 100,000 and 40,000 sites
CASES = [("periodic", (32, 32, 19)), ("periodic", (33, 31, 20)),
         ("lid", (43, 43, 42)), ("lid", (43, 43, 43)), ("lid", (250, 160, 2)), ("open", (43, 43, 43)),
         ("print", (46, 47, 46)), ("print", (47, 47, 46)),
         ("print2d", (199, 1, 201)), ("print2d", (201, 1, 200)), ("lid", (80001, 1, 1))]


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("kind,shape", CASES, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_stream_forms(kind, shape, storage):
    nx, ny, nz = shape
    if kind.startswith("print"):
        wl = I.print_run(shape, 4.0, 8, 0.03, 0.03, 0.6, storage, head_pos=(nx / 3.0 + 0.3, ny / 2.0 - 0.2 if ny > 1 else 0.0))
        if kind == "print2d":
            wl["params"] = dict(wl["params"], velset=O.D2Q9)
        init = None
    else:
        geom = {"periodic": dict(nozzle=0, z_mode=O.Z_PERIODIC),
                "lid": dict(nozzle=0, z_mode=O.Z_WALLS, top_mode=O.TOP_WALL, top_vel=(0.02, 0.01, 0.0)),
                "open": dict(nozzle=0, z_mode=O.Z_WALLS, top_mode=O.TOP_OPEN, rho_top_amb=1.01)}[kind]
        wl = dict(params=dict(velset=O.D3Q19, storage=storage, A=0.02, beta=0.7, tau_amb=0.9), geom=geom,
                  rheo=dict(law=O.POWER_LAW, n=0.6, K=0.05, tau_min=0.51, tau_max=2.0))
        rY, rB = I.droplet(shape, (0.4 * nx, 0.5 * ny, 0.6 * nz), 0.3 * min(nx, 40, 4 * nz), width=1.2)
        z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
        u = 0.01 * np.stack([np.sin(2 * np.pi * y / 16 + 1), np.cos(2 * np.pi * x / 16), np.sin(2 * np.pi * x / 16 + 2)])
        init = f32_exact(rY, rB, u)
    fg, fo, _ = run_pair(shape, wl, 6, "plain", storage=storage, init=init)
    tol, names = BARS[storage]
    if kind == "print2d":
        names = tuple(k for k in names if k != "uy")
    assert_close(fg, fo, tol, names=names, label="%s %s %s" % (kind, shape, storage))
