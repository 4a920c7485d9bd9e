"""Checkpoint files: the state comes back whole at the edges of strips and of the
part of the file that is converted at a time, and the host holds it once."""
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_common import oracle_case, slab_fields

pytestmark = pytest.mark.gpu

PROGRAM = """
import os, resource, sys
import numpy as np
from paper_2106_01557_gb300 import lbm
lat = lbm.Lattice.create(1024, 2048, precision="f64")
p = lat.params()
one = np.ones((2048, 1024))
lat.set_fields(p["rho_v"] * one, 0 * one, 0 * one, p["T0"] * one)
path = sys.argv[1]

def rss():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

def peak():
    return resource.getrusage(resource.RUSAGE_SELF).ru_maxrss * 1024

for call in (lat.save, lat.load):
    before = rss()
    reached = peak()
    call(path)
    size = os.path.getsize(path)
    # the file, and what the library allocates beside it
    assert peak() <= max(reached, before + 1.25 * size), (call, (peak() - before) / size)
"""


def test_peak_host_memory(gpu_lib, tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM, str(tmp_path / "state")], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr


OPTS = [{}, dict(walls=1, accel_y=-1e-5, Tr_bottom=0.8, Tr_hot=0.95, hot_x0=3, hot_len=4), dict(walls=1, open_sides=15, Tr_open=0.85)]


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("opts", OPTS, ids=["periodic", "walls", "open"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 40), (64, 9), (65, 33), (200, 17)])  # (8 x 8: the file is longer than the scratch area)
def test_resumed_state_is_the_saved_one(gpu_lib, tmp_path, nx, ny, opts, prec):
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny, **opts)
    rho, ux, uy, T = slab_fields(o, seed=3, eps=0.01, uamp=0.005)
    if "open_sides" in opts:
        rho = np.full_like(rho, o.p.rho_v)
    a, b = (lbm.Lattice.create(nx, ny, precision=prec, **opts) for _ in range(2))
    a.set_fields(rho, ux, uy, T)
    b.set_fields(rho * 0.9, ux, uy, T)  # another state, in the other buffer
    b.step(1)
    a.step(3)
    a.save(str(tmp_path / "a"))
    b.load(str(tmp_path / "a"))
    b.save(str(tmp_path / "b"))
    assert (tmp_path / "a").read_bytes() == (tmp_path / "b").read_bytes() and b.steps == 3
    for lat in (a, b):
        lat.step(4)
    assert all(np.array_equal(x, y) for x, y in zip(a.get_populations(), b.get_populations()))
    assert np.array_equal(a.step_stats(), b.step_stats())
