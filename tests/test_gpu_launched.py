"""The two launched step kernels against the FP64 oracle on lattices small enough
for the one launch they take by default: direct launches and replayed graphs of
a length that is not the default.

Tolerances as in test_gpu_parity.py for the same geometries: rel-L2 of rho and u
1e-10 (FP64) and 1e-5 (FP32) after 1000 steps, populations 1e-13 on random
geometries in FP64.
"""
import numpy as np
import pytest

import lbm_inputs as I
from lbm_pair import make_pair, rel_l2

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-10, "f32": 1e-5}


@pytest.mark.parametrize("tube", ["short", "bulk"])
@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("wall_model", [1, 0])
def test_tubes_1000_steps(storage, wall_model, tube):
    geo, kappa = ((I.tube(8, 64, u_mean=0.025), 12.0) if tube == "short" else
                  (I.tube(12, 159, u_mean=0.025), 18.0))
    lat, orc = make_pair(geo, storage, tau=0.8, wall_model=wall_model, F=0.85, kappa=kappa)
    lat.tune(graph_steps=50 if tube == "bulk" else 0)
    lat.step(1000)
    lat.sync()
    orc.run(1000)
    for a, b in zip(lat.moments(), orc.moments()):
        assert rel_l2(a, b) <= TOL[storage]
    for a, b in zip(lat.wall_state(), orc.wall_state()) if wall_model else ():
        assert rel_l2(a, b) <= 10 * TOL[storage]


@pytest.mark.parametrize("seed,shape", [(0, (8, 8, 8)), (1, (13, 9, 17)), (3, (33, 17, 9)),
                                        (4, (14, 11, 3))])
@pytest.mark.parametrize("wall_model", [1, 0])
def test_random_geometries_f64(seed, shape, wall_model):
    geo = I.random_labels(seed, shape, fill=0.75)
    lat, orc = make_pair(geo, "f64", tau=0.9, wall_model=wall_model, F=0.5, kappa=3.0,
                         rho0=0.999, fields=I.random_fields(seed, shape, drho=1e-3, umax=0.02))
    lat.tune(graph_steps=2 if seed & 1 else 0)
    for chunk in (1, 2, 17):
        lat.step(chunk)
        orc.run(chunk)
        np.testing.assert_allclose(lat.populations(), orc.populations(), rtol=0, atol=1e-13)
