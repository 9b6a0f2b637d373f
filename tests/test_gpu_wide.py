"""A periodic FP32 lattice with more tile rows than a launch has in y: it runs the
phase-by-phase kernels, as path "plain" does."""
import numpy as np
import pytest

from test_gpu_parity import _lbm, f32_exact

pytestmark = pytest.mark.gpu


def test_periodic_lattice_with_more_tile_rows_than_a_launch():
    lbm = _lbm()
    shape = (2, 8 * 65535 + 1, 3)
    nx, ny, nz = shape
    y = np.broadcast_to(np.arange(ny)[None, :, None], (nz, ny, nx))
    c = 0.5 * (1.0 + np.sin(2 * np.pi * y / 23.0))
    init = f32_exact(c, 1.0 - c)
    outs = []
    for path in ("auto", "plain"):
        lat = lbm.Lattice(shape, dict(velset=1, storage="f32", A=0.02, beta=0.7, tau_amb=0.9), dict(nozzle=0, z_mode=0),
                          dict(law=2, n=0.6, K=0.05, tau_min=0.51, tau_max=2.0), path=path)
        lat.set_fields(*init)
        lat.step(3)
        outs.append({k: v for k, v in lat.fields().items() if k != "diag"})
        lat.close()
    for k in outs[0]:
        assert np.array_equal(outs[0][k], outs[1][k]), k
    assert np.abs(np.asarray(outs[0]["uy"])).max() > 0
