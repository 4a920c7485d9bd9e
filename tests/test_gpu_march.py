"""The row-marching step at the edges of its strips (32 nodes, 64 for 16-bit
storage), blocks (4 strips) and chunks of rows, against the FP64 oracle."""
import struct

import numpy as np
import pytest

from gpu_common import gpu_case, oracle_case, rel_err, slab_fields
from paper_2106_01557_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = 7
# FP64 and FP32: the parity bounds of the suite. 16-bit storage rounded to
# nearest: every step rounds every population once, to 2^-11 (FP16) or 2^-8
# (BF16) of its size, so after n steps at most n times that of the largest.
TOL = {"f64": 1e-12, "f32": 1e-5, "f16s": STEPS * 2.0**-11, "bf16s": STEPS * 2.0**-8}
SIZES = [(8, 8), (31, 9), (32, 8), (33, 13), (63, 10), (64, 8), (65, 11), (127, 9), (129, 8), (257, 21)]
WALLS = dict(walls=1, accel_y=-1e-5, Tr_bottom=0.8, Tr_hot=0.95, hot_x0=3, hot_len=4)
OPEN = dict(walls=1, open_sides=15, Tr_open=0.85)


def _fields(o, opts):
    rho, ux, uy, T = slab_fields(o, seed=31, eps=0.01, uamp=0.005)
    if "open_sides" in opts:
        # vapour: the open sides next to a liquid a few nodes away drive the
        # oracle itself to negative temperatures
        rho = inputs.perturbed(np.full((o.ny, o.nx), o.p.rho_v), 0.01, 32)
    return rho, ux, uy, T


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("opts", [{}, WALLS, OPEN], ids=["periodic", "walls", "open"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_strip_edges_match_oracle(gpu_lib, nx, ny, opts, prec):
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny, **opts)
    fields = _fields(o, opts)
    o.init_fields(*fields)
    o.step(STEPS)
    g = lbm.Lattice.create(nx, ny, precision=prec, rounding=0, **opts)
    g.set_fields(*fields)
    g.step(STEPS)
    f, gg = g.get_populations()
    assert rel_err(f, o.f) < TOL[prec] and rel_err(gg, o.g) < TOL[prec]


@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16s"])
def test_batch_strip_edges_match_oracle(gpu_lib, prec):
    from paper_2106_01557_gb300 import lbm
    b = lbm.Batch([lbm.default_config(nx, ny, precision=prec, rounding=0) for nx, ny in SIZES])
    ors = [oracle_case(nx, ny) for nx, ny in SIZES]
    for shape in (0, 1):
        b.select(shape, 1)
        for i, o in enumerate(ors):
            fields = slab_fields(o, seed=50 + i, eps=0.01, uamp=0.005)
            b.set_fields(i, *fields)
            o.init_fields(*fields)
            o.step(STEPS)
        b.step(STEPS)
        for i, o in enumerate(ors):
            f, g = b.get_populations(i)
            assert rel_err(f, o.f) < TOL[prec] and rel_err(g, o.g) < TOL[prec], (shape, SIZES[i])


def test_record_of_every_step_count(gpu_lib):
    # the record is combined by the next step, by the last block of the last
    # step, or after a captured graph of 20 steps: the record of the last step
    # is that of the state entering it, whichever way the call ended
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(65, 40)
    fields = slab_fields(o, seed=3)
    for n in (1, 2, 20, 21, 40, 43):
        a, b = (lbm.Lattice.create(65, 40, precision="f64") for _ in range(2))
        for lat in (a, b):
            lat.set_fields(*fields)
        a.step(n)
        b.step(n - 1)
        s, before = a.step_stats(), b.conservation()
        assert s[7] == n and a.steps == n
        assert s[0] == pytest.approx(before[0], rel=1e-12) and s[4] == pytest.approx(before[4], rel=1e-11)
        assert s[3] == pytest.approx(before[3], rel=1e-12) and s[5] == pytest.approx(before[5], rel=1e-9)


@pytest.mark.parametrize("prec,line", [("f64", 16), ("f32", 32), ("f16s", 64)])
def test_checkpoint_file_keeps_its_planes(gpu_lib, tmp_path, prec, line):
    # the file: magic, nx, ny, precision, walls, configuration hash, steps, then
    # 18 planes of node rows from -2 on, `line` elements before column 0
    nx, ny = 77, 21
    o = oracle_case(nx, ny)
    g = gpu_case(nx, ny, prec)
    g.set_fields(*slab_fields(o, seed=8))
    g.step(3)
    path = tmp_path / "state.ck"
    g.save(str(path))
    raw = path.read_bytes()
    assert struct.unpack_from("<4i", raw, 8)[:2] == (nx, ny) and struct.unpack_from("<q", raw, 32)[0] == 3
    dtype = {"f64": np.float64, "f32": np.float32, "f16s": np.float16}[prec]
    pitch = -(-(line + nx + 16 // dtype().itemsize) // line) * line
    nyp = max(ny, 32 if prec == "f16s" else 16) + 4
    planes = np.frombuffer(raw, dtype, offset=40).reshape(18, nyp, pitch).astype(np.float64)
    f, gg = g.get_populations()
    ex, ey = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    for p in range(18):
        i = p % 9
        pulled = planes[p, 2 - ey[i]:2 - ey[i] + ny, line - ex[i]:line - ex[i] + nx]
        want = (f if p < 9 else gg)[i]
        shift = (want - pulled)[0, 0]  # 16-bit storage holds deviations from the rest populations
        assert (shift == 0.0 or prec == "f16s") and np.allclose(pulled + shift, want, rtol=0, atol=1e-15 if prec == "f64" else 1e-7)


@pytest.mark.parametrize("ncases,hi", [(3, 16), (40, 300)])
def test_batch_work_lists_cover_every_row_once(gpu_lib, ncases, hi):
    """Fewer rows than warps, and runs of rows that cross cases, columns of 1 to 10 strips and what is left of them."""
    from paper_2106_01557_gb300 import lbm
    sides = np.random.default_rng(ncases).integers(8, hi, (ncases, 2)).tolist()
    cfgs = [lbm.default_config(nx, ny, precision="f32") for nx, ny in sides]
    b = lbm.Batch(cfgs)
    for shape in (0, 1):
        for order in (0, 1, 2):
            b.select(shape, order)
            for i, (c, (nx, ny)) in enumerate(zip(cfgs, sides)):
                o = oracle_case(nx, ny)
                b.set_fields(i, *slab_fields(o, seed=50 + i, eps=0.01, uamp=0.005))
            b.step(2)
            for i, (c, (nx, ny)) in enumerate(zip(cfgs, sides)):
                f, _ = b.get_populations(i)
                # the record sums each row's density once (FP32 sums)
                assert abs(b.step_stats(i)[0] / f.sum() - 1) < 1e-5, (shape, order, i)
                if shape == 0 and order == 0:
                    s = lbm.Lattice(c)
                    s.set_fields(*slab_fields(oracle_case(nx, ny), seed=50 + i, eps=0.01, uamp=0.005))
                    s.step(2)
                    want = s.get_populations()
                    s.close()
                    first = [want] if i == 0 else first + [want]
                assert all(rel_err(a, w) < 1e-5 for a, w in zip(b.get_populations(i), first[i])), (shape, order, i)


def _macro_close(m, o, c, tol):
    want = o.moments()
    want = want if isinstance(want, dict) else dict(zip(("rho", "ux", "uy", "T"), want))
    assert rel_err(m["rho"], want["rho"]) < tol and rel_err(m["T"], want["T"]) < tol
    assert all(np.abs(m[k] - want[k]).max() < tol * c for k in ("ux", "uy"))


# of the suite's parity bounds: initial populations in the arithmetic of the
# storage and rounded once, fields of the state as it is stored in the arithmetic
# alone (a batch computes both in FP64)
@pytest.mark.parametrize("prec", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("opts", [{}, WALLS, OPEN, dict(cubic=1)], ids=["periodic", "walls", "open", "cubic"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_fields_in_and_out_match_oracle(gpu_lib, nx, ny, opts, prec):
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny, **opts)
    fields = _fields(o, opts)
    o.init_fields(*fields)
    once = {"f64": 1e-12, "f32": 1e-5, "f16s": 2.0**-11, "bf16s": 2.0**-8}[prec]
    exact = 1e-12 if prec == "f64" else 1e-5
    handles = [(lbm.Lattice.create(nx, ny, precision=prec, rounding=0, **opts), (), exact)]
    if not opts and prec != "f64":
        handles.append((lbm.Batch([lbm.default_config(nx, ny, precision=prec, rounding=0)]), (0,), 1e-12))
    for h, i, tol in handles:
        o.init_fields(*fields)
        h.set_fields(*i, *fields)
        f, g = h.get_populations(*i)
        assert rel_err(f, o.f) < once and rel_err(g, o.g) < once
        o.set_populations(f, g)
        _macro_close(h.moments(*i), o, o.p.c, tol)
        got, want = h.conservation(*i), o.conservation()
        assert abs(got[0] / want[0] - 1) < tol and abs(got[3] / want[3] - 1) < tol and abs(got[5] - want[5]) < tol * o.p.c
        assert max(abs(got[1] - want[1]), abs(got[2] - want[2])) < tol * want[0] * o.p.c
        if "open_sides" not in opts:  # (the oracle's total energy takes the density beyond an open side for a wall's)
            assert abs(got[4] - want[4]) < tol * abs(want[3])


# 1, 2, 3, 5 and 6 strips, in blocks of 1 to 4 warps: the blocks that combine the
# record of the step before, and the last block, take its quantities in shares
@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-5), ("f16s", 1e-3)])
@pytest.mark.parametrize("nx,ny", [(20, 400), (64, 33), (96, 500), (160, 90), (320, 40)])
def test_record_of_narrow_lattices(gpu_lib, nx, ny, prec, tol):
    from paper_2106_01557_gb300 import lbm
    o = oracle_case(nx, ny)
    fields = slab_fields(o, seed=31, eps=0.01, uamp=0.005)
    for n in (1, 2, 21, 40):
        g, h = (lbm.Lattice.create(nx, ny, precision=prec) for _ in range(2))
        for lat in (g, h):
            lat.set_fields(*fields)
        g.step(n)
        for _ in range(n):
            h.step(1)
        got = g.step_stats()
        # the record of a step is that of the state it began with, whichever block adds it up
        assert np.array_equal(got, h.step_stats()) and got[7] == n
        f = g.get_populations()[0]
        assert abs(got[0] / f.sum() - 1) < tol
        g.close()
        h.close()
