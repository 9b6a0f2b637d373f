"""State storage against populations (path "plain"), both FP32, over 60 steps of
small print runs: its velocities are no further from the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2102_02655_gb300 import inputs as I

from test_gpu_parity import _lbm, f32_exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,r,gap", [((64, 32, 32), 4.0, 12), ((70, 40, 41), 5.0, 12)], ids=["64x32x32", "70x40x41"])
def test_velocities_no_further_from_the_oracle_than_with_populations(shape, r, gap):
    lbm = _lbm()
    sq = {"auto": 0.0, "plain": 0.0}
    for seed in range(1, 5):
        wl = I.print_run(shape, r, gap, 0.02, 0.03, 0.6, "f32", head_pos=(shape[0] / 3.0, shape[1] / 2.0))
        rY, rB = I.nozzle_fill(shape, wl["geom"])
        init = f32_exact(rY, I.perturbed_ambient(shape, rB, seed=seed))
        ref = O.Oracle(shape, params=wl["params"], geom=wl["geom"], rheo=wl["rheo"])
        ref.set_fields(*init)
        ref.step(60)
        fo = ref.fields()
        for path in sq:
            lat = lbm.Lattice(shape, wl["params"], wl["geom"], wl["rheo"], path=path)
            lat.set_fields(*init)
            lat.step(60)
            f = lat.fields()
            lat.close()
            sq[path] += sum(((np.asarray(f[k], dtype=np.float64) - fo[k]) ** 2).sum() for k in ("ux", "uy", "uz"))
    assert sq["auto"] <= sq["plain"], sq
