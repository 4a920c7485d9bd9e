"""What a wall reflects with 16-bit storage and stochastic rounding (the default),
after one step, against the FP64 oracle's step from the same populations: each
reflected population is formed in FP32 and rounded once, to nearest, so it is
within half a step of the format of the exact value, up to FP32 rounding (the
suite's parity bound, 1e-5 of the largest population)."""
import numpy as np
import pytest

from gpu_common import oracle_case, slab_fields

pytestmark = pytest.mark.gpu

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
WALLS = dict(walls=1, accel_y=-1e-5, Tr_bottom=0.8, Tr_hot=0.95, hot_x0=3, hot_len=5)
BITS = {"f16s": 11, "bf16s": 8}  # of the significand


def _planes(raw, prec, nx, ny):
    words = np.frombuffer(raw, np.uint16, offset=40)
    values = words.view(np.float16).astype(np.float64) if prec == "f16s" else \
        (words.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    pitch = -(-(64 + max(nx, 64) + 8) // 64) * 64  # 64 elements before column 0, 16 bytes of ghosts, whole lines
    return values.reshape(18, max(ny, 32) + 4, pitch)


@pytest.mark.parametrize("prec", ["f16s", "bf16s"])
@pytest.mark.parametrize("opts", [WALLS, dict(walls=1, Tr_top=0.85)], ids=["hot-segment", "heated-top"])
@pytest.mark.parametrize("nx,ny", [(31, 9), (65, 11), (129, 8)])
def test_reflections_are_rounded_once(gpu_lib, tmp_path, nx, ny, opts, prec):
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny, **opts)
    lat = lbm.Lattice.create(nx, ny, precision=prec, **opts)
    lat.set_fields(*slab_fields(o, seed=17, eps=0.01, uamp=0.005))
    lat.step(3)
    o.set_populations(*lat.get_populations())
    o.step(1)
    lat.step(1)
    path = tmp_path / "state"
    lat.save(str(path))
    planes = _planes(path.read_bytes(), prec, nx, ny)
    got = lat.get_populations()
    for d, exact in enumerate((o.f, o.g)):
        for y, dirs in ((0, (2, 5, 6)), (ny - 1, (4, 7, 8))):
            for i in dirs:  # pulled from the ghost row: the reflections
                stored = planes[9 * d + i, y - EY[i] + 2, 64 - EX[i]:64 - EX[i] + nx]
                value = got[d][i, y]
                assert np.ptp(value - stored) < 1e-6  # (deviations from the rest populations)
                half = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(stored), 2.0**-14))) - BITS[prec])
                err = np.abs(value - exact[i, y])
                assert (err <= half + 1e-5 * np.abs(exact).max()).all(), (d, i, y, (err / half).max())


STEPS = 7


@pytest.mark.parametrize("prec", ["f16s", "bf16s"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (31, 9), (65, 11), (129, 8)])
def test_walled_steps_match_oracle(gpu_lib, nx, ny, prec):
    # stochastic rounding moves a value by less than one step of the format (2^-10 or
    # 2^-7 of its size), once per step: after n steps by at most n times that of the
    # largest population
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny, **WALLS)
    lat = lbm.Lattice.create(nx, ny, precision=prec, **WALLS)
    fields = slab_fields(o, seed=31, eps=0.01, uamp=0.005)
    o.init_fields(*fields)
    lat.set_fields(*fields)
    o.step(STEPS)
    lat.step(STEPS)
    for got, want in zip(lat.get_populations(), (o.f, o.g)):
        assert np.abs(got - want).max() < STEPS * 2.0 ** (1 - BITS[prec]) * np.abs(want).max()
