"""The one launch of small lattices belongs to the default knobs: a refused
lbm_tune, a knob set to its default, or set back to it, keeps it, another value
takes the launched kernels, and the autotuner times it as what it starts from.

Which of the two ran shows in the device bytes held: launched steps replay a
graph, whose step counter is allocated on first use.
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu


def _lat(storage="f32"):
    from paper_2108_08783_gb300 import Lattice
    geo = I.tube(7.5, 60, u_mean=0.02, u_amp=0.01, period=37.0)
    lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=0.75)
    lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=6.0)
    return lat


def _launched(lat):
    """Whether 40 more steps take the launched kernels, on a lattice that never did."""
    before = lat.info()[10]
    lat.step(40)
    lat.sync()
    return bool(lat.info()[10] != before)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s"])
def test_defaults_keep_the_one_launch(storage):
    from paper_2108_08783_gb300._capi import LbmError
    from paper_2108_08783_gb300.lattice import default_knobs
    lat = _lat(storage)
    assert not _launched(lat)
    for bad in (dict(bulk_warps=5), dict(prefetch=-1), dict(bulk_sites=6), dict(graph_steps=3)):
        with pytest.raises(LbmError):
            lat.tune(**bad)
    assert lat._lib.lbm_tune(lat.h, 99, 0) != 0
    assert not _launched(lat)
    lat.tune(graph_steps=20, **default_knobs(storage))
    assert not _launched(lat)
    lat.tune(bulk_warps=8)
    lat.tune(bulk_warps=4)
    assert not _launched(lat)
    lat.tune(bulk_warps=8)
    assert _launched(lat)
    lat.close()


def test_autotune_starts_from_the_one_launch():
    a, b = _lat(), _lat()
    held = a.info()[10]
    best, _ = a.autotune(bulk_sites=(1,), bulk_warps=(4,), prefetch=(4096,), graph_steps=(20,))
    assert best == dict(bulk_sites=1, bulk_warps=4, prefetch=4096, graph_steps=20)
    assert a.info()[10] == held
    b.step(a.step_count)
    np.testing.assert_array_equal(a.populations(), b.populations())
