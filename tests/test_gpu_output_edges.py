"""Output kernels at the edges of their blocks: lattices of one site, around a
warp's 32 and a block's 128, and irregular ones, after an even and an odd number
of steps.  Populations and moments against the FP64 oracle (1e-13, the bound of
the parity tests on such geometries), the density alone bit for bit that of the
full call, and nothing written beyond the last site.
"""
import ctypes as C

import numpy as np
import pytest

import lbm_inputs as I
from lbm_pair import make_pair

pytestmark = pytest.mark.gpu

GEOS = {"1": lambda: I.closed_box(3, 3, 3), "31": lambda: I.closed_box(3, 3, 33),
        "33": lambda: I.closed_box(3, 3, 35), "127": lambda: I.closed_box(3, 3, 129),
        "128": lambda: I.closed_box(3, 3, 130), "129": lambda: I.closed_box(3, 3, 131),
        "random": lambda: I.random_labels(3, (13, 9, 17), fill=0.75)}


@pytest.mark.parametrize("name", sorted(GEOS))
def test_outputs_match_the_oracle_and_stay_in_bounds(name):
    import torch
    geo = GEOS[name]()
    lat, orc = make_pair(geo, "f64", tau=0.9, wall_model=1, F=0.5, kappa=3.0, rho0=0.999,
                         fields=I.random_fields(2, geo.shape, drho=1e-3, umax=0.02))
    n = lat.n

    def buf(count):
        return torch.full((count + 64,), 7.0, dtype=torch.float64, device="cuda")

    for steps in (0, 1, 2, 3):  # before the first, then odd, odd and even counts
        lat.step(steps)
        orc.run(steps)
        f, rho, u, rho1 = buf(19 * n), buf(n), buf(3 * n), buf(n)
        ptr = [C.c_void_p(b.data_ptr()) for b in (f, rho, u, rho1)]
        lat._check(lat._lib.lbm_get_populations(lat.h, ptr[0], 1))
        lat._check(lat._lib.lbm_moments(lat.h, ptr[1], ptr[2], 1))
        lat._check(lat._lib.lbm_moments(lat.h, ptr[3], None, 1))
        lat.sync()
        for b, count in ((f, 19 * n), (rho, n), (u, 3 * n), (rho1, n)):
            assert bool((b[count:] == 7.0).all())
        assert torch.equal(rho, rho1)
        ro, uo = orc.moments()
        np.testing.assert_allclose(f[:19 * n].cpu().numpy().reshape(n, 19), orc.populations(),
                                   rtol=0, atol=1e-13)
        np.testing.assert_allclose(rho[:n].cpu().numpy(), ro, rtol=0, atol=1e-12)
        np.testing.assert_allclose(u[:3 * n].cpu().numpy().reshape(n, 3), uo, rtol=0, atol=1e-12)
