"""Print runs whose nozzle stands one to three sites above the substrate, so that
the nozzle box reaches plane 0 and its collision reads the substrate's ghost
plane: the fused path, alone and in a batch, against the oracle, on a lattice
wider than the box and with ink on the substrate across the box's edges. The
first head position puts the box's low side a whole number of sites from the
wall. (nu stays out for FP32: see test_gpu_parity.)"""
import numpy as np
import pytest

import oracle as O
from paper_2102_02655_gb300 import inputs as I

from test_gpu_parity import FIELDS, TOL, _lbm, assert_close, f32_exact
from test_gpu_storage16 import HYDRO, TOL16

pytestmark = pytest.mark.gpu

SHAPE = (40, 37, 16)
BARS = {"f64": (TOL["f64"], FIELDS), "f32": (TOL["f32"], tuple(k for k in FIELDS if k != "nu")), "f16dev": (TOL16, HYDRO)}


def _case(storage, gap, pos):
    wl = I.print_run(SHAPE, 3.0, gap, 0.03, 0.03, 0.6, storage, head_pos=pos)
    nx, ny, nz = SHAPE
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    layer = 0.5 * (1 - np.tanh((z - 2.0 - np.sin(2 * np.pi * x / nx) - np.cos(2 * np.pi * y / ny)) / 1.2))
    c = np.maximum(layer, I.nozzle_fill(SHAPE, wl["geom"])[0])
    rho = I.perturbed_ambient(SHAPE, np.ones_like(c), seed=3)
    return wl, f32_exact(c * rho, (1.0 - c) * rho)


@pytest.mark.parametrize("pos", [(13.0, 18.0), (13.4, 18.3)], ids=["whole", "between"])
@pytest.mark.parametrize("gap", [1, 2, 3])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
def test_box_on_the_substrate(storage, gap, pos):
    lbm = _lbm()
    wl, init = _case(storage, gap, pos)
    ref = O.Oracle(SHAPE, params=wl["params"], geom=wl["geom"], rheo=wl["rheo"])
    lats = [lbm.Lattice(SHAPE, wl["params"], wl["geom"], wl["rheo"], path="fused") for _ in range(2)]
    for m in [ref] + lats:
        m.set_fields(*init)
    batch = lbm.Batch(lats[1:])
    ref.step(30)
    lats[0].step(30)
    batch.step(30)
    tol, names = BARS[storage]
    fo = ref.fields()
    for label, lat in zip(("alone", "batch"), lats):
        assert_close(lat.fields(), fo, tol, names=names, label="%s gap %d %s" % (storage, gap, label))
    batch.close()
    for lat in lats:
        lat.close()
