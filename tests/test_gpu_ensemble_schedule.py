"""Ensemble: a refused schedule leaves the numbering of the tiles as it was, and a
change of schedule needs no device memory (it would fail half-way without any).

Members of different sizes (odd and even numbers of bulk tiles), relaxation times
and walls, stepped alone as the reference; the tolerance is the rounding level
of the other ensemble tests.
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,atol", [("f64", 1e-13), ("f32", 1e-6)])
def test_schedules_refused_and_without_device_memory(storage, atol):
    from paper_2108_08783_gb300 import Ensemble, Lattice
    from paper_2108_08783_gb300._capi import LbmError
    geos = [I.tube(r, n, u_mean=0.02, u_amp=0.01, period=300.0, phase=0.3 * k)
            for k, (r, n) in enumerate(((5.0, 70), (7.3, 120), (6.0, 65), (9.0, 200)))]
    alone, batch = ([Lattice(g.labels, g.iolets, storage=storage, tau=0.7 + 0.1 * k)
                     for k, g in enumerate(geos)] for _ in range(2))
    for lats in (alone, batch):
        for k, lat in enumerate(lats):
            lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=5.0 + k)
    ens = Ensemble(batch)

    def refused(value):
        with pytest.raises(LbmError):
            ens.tune(schedule=value)

    def no_memory(value):
        torch, batch[0]._alloc.torch = batch[0]._alloc.torch, None  # every allocation fails
        try:
            ens.tune(schedule=value)
        finally:
            batch[0]._alloc.torch = torch

    for change in (lambda: None, lambda: refused(7), lambda: no_memory(1), lambda: refused(-1),
                   lambda: no_memory(0)):
        change()
        ens.step(5)
        ens.sync()
        for a, b in zip(alone, batch):
            a.step(5)
            a.sync()
            np.testing.assert_allclose(b.populations(), a.populations(), rtol=0, atol=atol)
    ens.close()
