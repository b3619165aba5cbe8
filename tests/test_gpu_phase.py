"""The FP64 inlet's phase after very many steps: whole periods later, the same
populations give the same step.

T = 100,003 steps (no dyadic 1 / T), 10^7 periods later (10^12 steps). A phase
held to 2^-64 of a period and rounded to the nearest FP64 number of half periods
errs by at most 2e-16 rad on either side; the inlet velocity, 0.05 at most, by
2e-17, and its populations, all below 0.1, by that and a rounding of 7e-18 in
each of a few operations: 2e-16 in all. An increment truncated to 2^-64 drifts
by up to 10^12 2^-64 periods, 3e-7 rad.
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launched", [False, True])
@pytest.mark.parametrize("m", [0, 12345])
def test_whole_periods_later_is_the_same_step(m, launched):
    from paper_2108_08783_gb300 import Lattice
    T = 100003
    out = []
    for step in (m, m + T * 10 ** 7):
        geo = I.tube(6, 20, u_mean=0.0, u_amp=0.05, period=float(T), phase=0.7)
        lat = Lattice(geo.labels, geo.iolets, storage="f64", tau=0.8)
        if launched:
            lat.tune(graph_steps=0)
        lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=6.0)
        f = lat.populations()
        lat.set_populations(f, step=step)
        lat.step(2)
        lat.sync()
        assert lat.step_count == step + 2
        out.append(lat.populations())
    assert np.abs(out[0] - f).max() > 1e-4  # the inlet acts
    assert np.abs(out[1] - out[0]).max() <= 2e-16
