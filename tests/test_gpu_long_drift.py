"""Mass over long runs: the collision and its back-transform keep it up to their
roundings, which must not share a bias. The model's runs of 100,000 steps drift by
1.7e-5 (FP32), 1.3e-13 (FP64) and, with stochastic rounding, 8e-5 (FP16S, whose
random part is about 3e-5 for a 1024 x 1024 lattice); the bounds are twice that
(FP16S three times, mean of four runs), in proportion to the steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _drift(n, prec, steps, seed):
    from paper_2106_01557_gb300 import inputs, lbm
    lat = lbm.Lattice.create(n, n, precision=prec)
    p = lat.params()
    rho = inputs.perturbed(inputs.slab(n, n, p["rho_v"], p["rho_l"], n / 4, 3 * n / 4, 4.0), 0.01, seed)
    z = 0 * rho
    lat.set_fields(rho, z, z, z + p["T0"])
    lat.step(2000)
    before = lat.conservation()[0]
    lat.step(steps)
    after = lat.conservation()[0]
    lat.close()
    return after / before - 1


@pytest.mark.parametrize("prec,n,steps,runs,bound", [("f64", 512, 20000, 1, 2 * 1.3e-18), ("f32", 1024, 40000, 1, 2 * 1.7e-10),
                                                     ("f16s", 1024, 60000, 4, 3 * 8e-10)])
def test_mass_drift(gpu_lib, prec, n, steps, runs, bound):
    drift = float(np.mean([_drift(n, prec, steps, seed) for seed in range(runs)]))
    assert abs(drift) < bound * steps, drift
