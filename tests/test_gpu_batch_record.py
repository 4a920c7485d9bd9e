"""The record of a batch is as exact for tall boxes as for flat ones: FP32 sums
cover 16 rows of a strip, FP64 sums from there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# roundings of an FP32 sum: 15 additions of rows, one of the two nodes of a lane
# (16-bit storage), five over the lanes; each at most 2^-24 of the sum
BOUND = 21 * 2.0**-24


def _records(nx, ny, densities, prec):
    from paper_2106_01557_gb300 import lbm
    b = lbm.Batch([lbm.default_config(nx, ny, precision=prec, rounding=0) for _ in densities])
    T, z = np.full((ny, nx), b.params(0)["T0"]), np.zeros((ny, nx))
    for i, r in enumerate(densities):
        b.set_fields(i, np.full((ny, nx), r), z, z, T)
    b.step(1)
    out = np.array([b.step_stats(i) for i in range(len(densities))])
    b.close()
    return out[:, [0, 3, 4]] / (nx * ny)


@pytest.mark.parametrize("prec,nx", [("f16s", 1216), ("f32", 608)])
def test_record_of_tall_boxes(gpu_lib, prec, nx):
    # Uniform boxes, whose roundings do not average out, in runs of 500 rows per warp
    # on 152 multiprocessors; the same states in boxes of one row per warp. (With
    # FP32 sums over 500 rows the two differ by up to 7e-6.)
    densities = np.linspace(0.05, 0.35, 16)
    tall = _records(nx, 2000 if prec == "f16s" else 4000, densities, prec)
    flat = _records(64, 16, densities, prec)
    assert np.abs(tall / flat - 1).max() < 2 * BOUND
