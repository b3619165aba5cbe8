"""Small lattices: all steps of a call in one launch (a warp per tile, a grid
barrier between steps), against the two launched kernels of every step, which
setting a launch knob selects. Both inline the same updates with every
operation written out, so populations and wall state are equal bit for bit.

Sizes: one site; one tile less, exactly and one more than full; every kind of
tile (bulk, coherent, irregular with few and with many runs); around the most
tiles the one launch takes (16 per SM); and a lattice with sites linked to two
iolets, which always takes the launched kernels. Step counts: one, odd and
even, with diagnostic steps between, and more than one launch holds.
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

GEOMETRIES = {
    "one_site": lambda: I.closed_box(3, 3, 3),
    "31": lambda: I.closed_box(3, 3, 33),
    "32": lambda: I.closed_box(3, 3, 34),
    "33": lambda: I.closed_box(3, 3, 35),
    "tube": lambda: I.tube(7.5, 150, u_mean=0.02, u_amp=0.01, period=37.0),
    "random": lambda: I.random_labels(1, (17, 15, 21)),
    "tree": lambda: I.murray_tree(seed=3, depth=2, root_radius=7.0),
    "two_iolets": lambda: I.random_labels(4, (14, 11, 3)),
}


def _pair(geo, storage, wall="elastic"):
    from paper_2108_08783_gb300 import Lattice
    lats = []
    for launched in (False, True):
        lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=0.75)
        lat.set_wall(wall, rho0=1.0, F=0.85, kappa=6.0)
        if launched:
            lat.tune(graph_steps=0)
        c = lat.coords()
        rho, u = I.random_fields(2, geo.shape)
        lat.init_fields(I.gather(rho, c), I.gather(u, c))
        lats.append(lat)
    return lats


def _equal(a, b):
    a.sync()
    b.sync()
    assert a.step_count == b.step_count
    np.testing.assert_array_equal(a.populations(), b.populations())
    for x, y in zip(a.wall_state(), b.wall_state()):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
@pytest.mark.parametrize("name", sorted(GEOMETRIES))
def test_one_launch_equals_launched_steps(name, storage):
    geo = GEOMETRIES[name]()
    if geo.iolets and geo.iolets[0].u_mean == 0.0:
        geo.iolets[0].u_mean = 0.01
    for wall in ("elastic", "bounceback"):
        a, b = _pair(geo, storage, wall)
        for n in (1, 2, 7, 24):
            a.step(n)
            b.step(n)
        _equal(a, b)
        da, db = a.step_diag(4), b.step_diag(4)
        a.step(3)
        b.step(3)
        _equal(a, b)
        np.testing.assert_array_equal(da, db)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_largest_small_lattice_and_the_next(storage):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for planes in (sms, sms + 1):  # planes of 8 x 64 sites: 16 tiles each
        geo = I.closed_box(2 + planes, 10, 66)
        a, b = _pair(geo, storage)
        for k in (1, 6):
            a.step(k)
            b.step(k)
        _equal(a, b)


def test_more_steps_than_one_launch_and_another_stream():
    import ctypes as C

    import torch
    geo = I.tube(5, 40, u_mean=0.01)
    a, b = _pair(geo, "f32")
    a.step(2345)
    b.step(2345)
    _equal(a, b)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    a._check(a._lib.lbm_set_stream(a.h, C.c_void_p(s.cuda_stream)))
    a.step(11)
    b.step(11)
    _equal(a, b)
