"""Output kernels (moments, populations) on both population layouts and on
sizes at the edges of the 32-site tiles and the 128-site blocks, with a
lattice whose tiles are bulk, coherent and irregular.

``moments`` must agree with the sums over ``populations`` of the same state:
both read the same stored values, so the difference is rounding alone.  FP64
storage: 19 additions of values below 1 (19 * 2^-53 relative, and the same
for the momentum and the division): 1e-14.  The others form rho - 1 and
rho u from g in FP32: at most 19 roundings of partial sums below 0.2, i.e.
19 * 0.2 * 2^-24 = 2.3e-7 absolute, and as much again in u = j / rho.
"""
import ctypes as C

import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

GEOMETRIES = {
    "one_site": lambda: I.closed_box(3, 3, 3),
    "tile_31": lambda: I.closed_box(3, 3, 33),
    "tile_32": lambda: I.closed_box(3, 3, 34),
    "block_129": lambda: I.closed_box(3, 5, 45),
    "tube_bulk": lambda: I.tube(9, 131, u_mean=0.02),
    "random": lambda: I.random_labels(3, (13, 11, 17)),
}


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("name", sorted(GEOMETRIES))
def test_moments_are_the_sums_of_the_populations(name, storage):
    import torch
    from paper_2108_08783_gb300 import Lattice
    geo = GEOMETRIES[name]()
    lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=0.8)
    lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=4.0)
    rho, u = I.random_fields(1, geo.shape)
    c = lat.coords()
    lat.init_fields(I.gather(rho, c), I.gather(u, c))
    vel = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1],
                    [0, 0, -1], [1, 1, 0], [-1, -1, 0], [1, -1, 0], [-1, 1, 0], [1, 0, 1],
                    [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1],
                    [0, -1, 1]], float)
    tol = 1e-14 if storage == "f64" else 5e-7
    for steps in (0, 1, 1):  # even, odd, even layout
        lat.step(steps)
        f = lat.populations()
        rho_f = f.sum(1)
        u_f = f @ vel / rho_f[:, None]
        # guard elements behind the outputs stay as they are
        r = torch.full((lat.n + 32,), 7.0, dtype=torch.float64, device="cuda")
        w = torch.full((3 * lat.n + 96,), 7.0, dtype=torch.float64, device="cuda")
        lat.moments_into(r[:lat.n], w[:3 * lat.n].view(-1, 3))
        lat.sync()
        r, w = r.cpu().numpy(), w.cpu().numpy()
        assert np.all(r[lat.n:] == 7.0) and np.all(w[3 * lat.n:] == 7.0)
        assert np.abs(r[:lat.n] - rho_f).max() <= tol
        assert np.abs(w[:3 * lat.n].reshape(-1, 3) - u_f).max() <= tol
        # either output alone
        only = torch.zeros(lat.n, dtype=torch.float64, device="cuda")
        lat._check(lat._lib.lbm_moments(lat.h, C.c_void_p(only.data_ptr()), None, 1))
        lat.sync()
        assert np.array_equal(only.cpu().numpy(), r[:lat.n])
        # populations set and read back survive unchanged in this layout
        lat.set_populations(f, int(lat.info()[7]))
        assert np.array_equal(lat.populations(), f)
