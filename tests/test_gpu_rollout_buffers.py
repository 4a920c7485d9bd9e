"""A surrogate handle rolls out on lattices of any size one after another: the
fields of a rollout are sized by nodes, its snapshot by the bytes of the state,
which are not in proportion (a 16 x 1000 lattice in FP64 has more bytes than a
256 x 256 one in FP32, and a fourth of its nodes)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_rollout_on_a_larger_lattice_of_fewer_bytes(gpu_lib):
    from oracle import Oracle, thermo
    from oracle import surrogate as S
    from paper_2106_01557_gb300 import inputs, lbm
    pp = Oracle(thermo.Config(nx=256, ny=256)).p
    p = S.init_params(channels=64, blocks=2, seed=0)
    p["proj"] = (0 * p["proj"][0], 0 * p["proj"][1])  # the prediction is the state itself
    params = lbm.surrogate_params_from_oracle_layout(p)

    def sur():
        s = lbm.Surrogate([pp.rho_v, 0.0, 0.0, pp.T0], [pp.rho_l - pp.rho_v, 0.01 * pp.c, 0.01 * pp.c, 0.05 * pp.Tc], K=10, blocks=2)
        s.set_params(params)
        return s

    def rollout(s, nx, ny, prec):
        rho = inputs.droplets(nx, ny, pp.rho_v, pp.rho_l, [(nx / 2, ny / 2)], [5], 4.0)
        lat = lbm.Lattice.create(nx, ny, precision=prec)
        lat.set_fields(rho, 0 * rho, 0 * rho, 0 * rho + pp.T0)
        st = s.rollout(lat, 2, verify_steps=2, field_tol=0.9)
        pops = lat.get_populations()
        lat.close()
        return {k: v for k, v in st.items() if not k.startswith("ms_")}, pops

    used, fresh = sur(), sur()
    rollout(used, 16, 1000, "f64")
    (a, fa), (b, fb) = rollout(used, 256, 256, "f32"), rollout(fresh, 256, 256, "f32")
    assert a == b and all(np.array_equal(x, y) for x, y in zip(fa, fb))
