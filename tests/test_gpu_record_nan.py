"""The record's largest speed with a node that is not a number: that of the others."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIVERGED = -4


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("ny", [8, 700])  # one row per warp, and runs of rows
def test_largest_speed_beside_a_nan(gpu_lib, prec, ny):
    from paper_2106_01557_gb300 import lbm
    lat = lbm.Lattice.create(64, ny, precision=prec, rounding=0)
    p = lat.params()
    one = np.ones((ny, 64))
    ux = 0.0 * one
    ux[4, 5] = 0.01 * p["c"]
    lat.set_fields(p["rho_v"] * one, ux, 0 * one, p["T0"] * one)
    f, g = lat.get_populations()
    lat.set_populations(f, g)
    lat.step(1)
    want = lat.step_stats()[5]
    assert want > 0.005 * p["c"]
    out = np.zeros(8)
    for x in range(9, 64):  # (the pair force takes it to the eight neighbours)
        h = f.copy()
        h[0, 4, x] = np.nan
        lat.set_populations(h, g)
        lat.step(1)
        rc = lat.lib.lbm_step_stats(lat.h, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
        assert rc == DIVERGED and out[6] > 0 and out[5] == want, x
