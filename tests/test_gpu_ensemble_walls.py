"""The ensemble's boundary kernel reads its tiles from descriptors, and takes the
wall model and "one F and kappa for the whole lattice" from the launch when all
members agree on them: members that agree, that differ in the wall model, in the
kind of their parameters (one value or one per wall site), changed between
calls, and an ensemble without any bulk tile, against the members stepped alone.

The two paths inline the same update with every operation spelled out; the
tolerance is the one of the other ensemble tests all the same (rounding level).
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

ATOL = {"f64": 1e-13, "f32": 1e-6, "f16s": 1e-4}


def _set(lat, kind):
    n = lat.n_wall
    if kind == "bounceback":
        lat.set_wall("bounceback", rho0=1.0)
    elif kind == "uniform":
        lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=9.0)
    else:
        k = np.arange(n)
        lat.set_wall("elastic", rho0=0.999, F=0.7 + 0.2 * (k % 7) / 7, kappa=2.0 + k % 5)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("sizes", [((5.0, 40), (7.3, 33), (6.0, 65)), ((2.0, 9), (2.5, 5), (3.0, 7))])
def test_walls_of_every_mix_equal_members_alone(storage, sizes):
    from paper_2108_08783_gb300 import Ensemble, Lattice
    geos = [I.tube(r, n, u_mean=0.02, u_amp=0.01, period=300.0, phase=0.3 * k)
            for k, (r, n) in enumerate(sizes)]
    alone, batch = ([Lattice(g.labels, g.iolets, storage=storage, tau=0.7 + 0.1 * k)
                     for k, g in enumerate(geos)] for _ in range(2))
    ens = Ensemble(batch)
    for mix in (("uniform",) * 3, ("uniform", "sites", "uniform"),
                ("bounceback", "uniform", "sites"), ("bounceback",) * 3):
        for a, b, kind in zip(alone, batch, mix):
            _set(a, kind)
            _set(b, kind)
        ens.step(7)
        ens.sync()
        for a, b in zip(alone, batch):
            a.step(7)
            a.sync()
            np.testing.assert_allclose(b.populations(), a.populations(), rtol=0,
                                       atol=ATOL[storage])
    ens.close()
