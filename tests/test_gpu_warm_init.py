"""A warm start sets, at every site, the populations of the fields that a forward
pass over all sites' features gives.

The features and the network's outputs are the library's own, so only the last
steps differ: the FP64 fields, restated with torch, and their rounding to FP32
populations (density and momentum sums of 19 FP32 values: 19 * 2^-24 of the
largest of them, 1/3 for the density's deviation and 1 for the velocity's).
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius,length", [(3.0, 5), (16.0, 150), (24.0, 449)])
def test_populations_are_those_of_the_proposed_fields(radius, length):
    import torch
    from paper_2108_08783_gb300 import MLP, Lattice, warm_frame
    geo = I.tube(radius, length, u_mean=0.02)
    lat = Lattice(geo.labels, geo.iolets, storage="f32", tau=0.8)
    lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=10.0)
    c = geo.meta["centre"]
    fr = warm_frame(centre=(c[0], c[1], 0.0), axis=(0.0, 0.0, 1.0), z0=0.5, length=length,
                    radius=radius, features=[0.5, -0.2, 1.0, 0.3, 0.2], rho_scale=2e-3, u_scale=0.02)
    net = MLP(7, 64, 3, 3, max_batch=256)
    net.set_params(I.mlp_init(1, 7, 64, 3, 3, bias_scale=0.2))
    x, _ = lat.warm_features(fr)
    y = net.forward(x)
    net.sync()
    y = y.double().cpu().numpy()
    for _ in range(2):  # over populations of zero, and over its own
        lat.warm_start(net, fr)
        rho, u = lat.moments()
        d = lat.coords()[:, :2] - np.array([c[0], c[1]])
        r = np.hypot(d[:, 0], d[:, 1])
        er = np.where(r[:, None] > 1e-12, d / np.maximum(r, 1e-300)[:, None], 0.0)
        ref = 0.02 * np.hstack([y[:, 1:2] * er, y[:, 2:3]])
        # 4e-6 of the velocities' scale adds the division by rho and FP32's own u
        assert np.abs(rho - (1 + 2e-3 * y[:, 0])).max() < 19 * 2.0 ** -24 * 0.4
        assert np.abs(u - ref).max() < 19 * 2.0 ** -24 + 4e-6 * np.abs(ref).max()
        lat.step(3)
        lat.sync()
