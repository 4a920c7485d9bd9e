"""The bound on a warp's wait for its first rows: one that no wait can meet is
reported, and the next state steps as if nothing had been."""
import numpy as np
import pytest

from gpu_common import oracle_case, slab_fields

pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s", "bf16s"])
def test_lattice(gpu_lib, prec):
    # 1 ns: no load returns in that time. (0 is answered before any load.)
    from paper_2106_01557_gb300 import lbm
    nx = ny = 300
    fields = slab_fields(oracle_case(nx, ny), seed=5)
    a, b = (lbm.Lattice.create(nx, ny, precision=prec) for _ in range(2))
    for lat in (a, b):
        lat.set_fields(*fields)
    a.set_tile_wait(1)
    a.step(1)
    with pytest.raises(lbm.LbmError) as e:
        a.synchronize()
    assert e.value.code == TIMEOUT
    a.set_tile_wait(2_000_000_000)
    a.set_fields(*fields)
    b.step(1)
    b.set_fields(*fields)  # (both have counted one step, which keys the rounding of 16-bit storage)
    for lat in (a, b):
        lat.step(5)
    assert all(np.array_equal(x, y) for x, y in zip(a.get_populations(), b.get_populations()))


@pytest.mark.parametrize("prec", ["f32", "f16s"])
def test_batch(gpu_lib, prec):
    from paper_2106_01557_gb300 import lbm
    sizes = [(200, 120), (64, 400), (130, 90)]
    a, b = (lbm.Batch([lbm.default_config(nx, ny, precision=prec) for nx, ny in sizes]) for _ in range(2))

    def reset(h):
        for i, (nx, ny) in enumerate(sizes):
            h.set_fields(i, *slab_fields(oracle_case(nx, ny), seed=9 + i))

    reset(a)
    reset(b)
    a.set_tile_wait(1)
    a.step(1)
    with pytest.raises(lbm.LbmError) as e:
        a.synchronize()
    assert e.value.code == TIMEOUT
    a.set_tile_wait(2_000_000_000)
    b.step(1)
    for h in (a, b):
        reset(h)
        h.step(5)
    for i in range(len(sizes)):
        assert all(np.array_equal(x, y) for x, y in zip(a.get_populations(i), b.get_populations(i)))
