"""The bulk kernels' shrinking plane chunks (taken where more CTAs than run at
once are launched: above 304 for the state kernel, 152 in FP64 and 456 in 16-bit
storage) change no bit, empty chunks among them; and the open top's ledger of the
state kernel agrees with the populations' and the oracle's."""
import numpy as np
import pytest

import oracle as O

from test_gpu_parity import _lbm
from test_gpu_state import _case

pytestmark = pytest.mark.gpu

SHAPE = (70, 66, 23)  # 3 x 9 tile columns: 621 CTAs at one plane a chunk


def _run(monkeypatch, shape, wl, init, storage, zchunk, path, steps):
    monkeypatch.setenv("CGLBM_ZCHUNK", str(zchunk))
    lat = _lbm().Lattice(shape, dict(wl["params"], storage=storage), wl["geom"], wl["rheo"], path=path)
    lat.set_fields(*init)
    lat.step(steps)
    f = lat.fields()
    lat.close()
    return f


@pytest.mark.parametrize("storage,z_mode", [("f32", O.Z_WALLS), ("f32", O.Z_PERIODIC), ("f64", O.Z_WALLS), ("f16dev", O.Z_WALLS)])
def test_shrinking_chunks_change_no_bit(monkeypatch, storage, z_mode):
    wl, init = _case(SHAPE, z_mode)
    one, many = (_run(monkeypatch, SHAPE, wl, init, storage, zc, "auto", 10) for zc in (SHAPE[2], 1))
    for k in one:
        if k != "diag":
            assert np.array_equal(one[k], many[k]), k
    assert np.allclose(one["diag"]["mass"], many["diag"]["mass"], rtol=1e-12)


def test_open_top_ledger_of_the_state_kernel(monkeypatch):
    """Sums of the same links from rounded populations: 1e-6 of the mass."""
    shape = (45, 19, 23)
    wl, init = _case(shape, O.Z_WALLS)
    ref = O.Oracle(shape, params=wl["params"], geom=wl["geom"], rheo=wl["rheo"])
    ref.set_fields(*init)
    ref.step(15)
    d = ref.diag()
    m = sum(d["mass"])
    assert np.abs(d["bc_flux"]).max() > 1e-4 * m
    for zc, path in ((23, "auto"), (8, "auto"), (1, "auto"), (23, "plain")):
        f = _run(monkeypatch, shape, wl, init, "f32", zc, path, 15)
        assert np.allclose(f["diag"]["bc_flux"], d["bc_flux"], rtol=0, atol=1e-6 * m), (zc, path)
