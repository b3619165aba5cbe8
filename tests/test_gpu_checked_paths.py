"""The checked build (-DLBM_CHECKED) over the step paths beside a lattice's two
launched kernels: all steps of a small lattice in one launch, and ensembles, in
every storage and pairing of the bulk kernels, with 4 and 8 warps per CTA and
with graphs and members of odd and even numbers of bulk tiles.

The same build takes the descending odd steps of populations beyond L2 on these
small ones (-DLBM_ALTERNATE_BYTES=0): ensembles, and single lattices' launched
kernels in every pairing (staged rows too), with uniform and per-site walls, sites linked to two
iolets, and diagnostic steps.

Neighbour indices are range-checked in all of them (LBM_ECHECK from the next
sync), the stores of the one launch are counted over its steps, and the fields
are those of the package's build, bit for bit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = r"""
import sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np
from test_gpu_checked_paths import run
np.savez(sys.argv[2], *run())
"""


def _lat(geo, storage, k=0, wall="elastic"):
    from paper_2108_08783_gb300 import Lattice
    lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=0.7 + 0.1 * k)
    lat.set_wall(wall, rho0=1.0, F=0.85, kappa=5.0 + k)
    rho, u = I.random_fields(2, geo.shape)
    c = lat.coords()
    lat.init_fields(I.gather(rho, c), I.gather(u, c))
    return lat


def _launched():
    """Single lattices through the two launched kernels of a step."""
    out = []
    geos = [I.tube(7.5, 255, u_mean=0.02, u_amp=0.01, period=37.0), I.closed_box(3, 3, 35),
            I.murray_tree(seed=3, depth=2, root_radius=7.0),
            I.random_labels(4, (14, 11, 3), fill=0.8)]  # sites linked to two iolets
    for storage in ("f32", "f16s", "bf16s"):
        for mode in (1, 2, 3, 4) if storage == "f32" else (1, 2, 3, 4, 5):
            for k, geo in enumerate(geos):
                for warps in (4, 8):
                    lat = _lat(geo, storage)
                    if warps == 8 and lat.n_wall:  # F and kappa of every wall site
                        w = np.arange(lat.n_wall)
                        lat.set_wall("elastic", rho0=1.0, F=0.7 + 0.02 * (w % 7),
                                     kappa=2.0 + w % 5)
                    lat.tune(bulk_sites=mode, bulk_warps=warps, graph_steps=0,
                             prefetch=(0, 3, 64, 4096)[k])
                    diag = []
                    for n in (1, 2, 2, 4):
                        lat.step(n)
                        diag.append(lat.step_diag(n))
                    lat.sync()
                    out += [lat.populations(), np.array(diag), *lat.wall_state()]
                    lat.close()
    return out


def run():
    from paper_2108_08783_gb300 import Ensemble
    out = _launched()
    geos = [I.tube(7.5, 150, u_mean=0.02, u_amp=0.01, period=37.0), I.closed_box(3, 3, 34),
            I.murray_tree(seed=3, depth=2, root_radius=7.0), I.random_labels(1, (17, 15, 21))]
    for storage in ("f64", "f32", "f16s", "bf16s"):
        for wall in ("elastic", "bounceback"):
            for geo in geos:
                lat = _lat(geo, storage, wall=wall)
                for n in (2, 5, 6):
                    lat.step(n)
                    lat.sync()
                out.append(lat.populations())
                lat.close()
    geos = [I.tube(7.5, 255, u_mean=0.02, u_amp=0.01, period=300.0, phase=0.3),
            I.murray_tree(seed=3, depth=2, root_radius=7.0),
            I.tube(7.3, 290, u_mean=0.02, u_amp=0.01, period=200.0), I.closed_box(7, 9, 290)]
    for storage in ("f64", "f32", "f16s", "bf16s"):
        for mode in (1,) if storage == "f64" else (1, 2, 3, 4):
            for warps in (4, 8):
                members = [_lat(g, storage, k) for k, g in enumerate(geos)]
                assert [int(m.info()[4]) & 1 for m in members] == [1, 1, 0, 1]
                ens = Ensemble(members)
                ens.tune(bulk_sites=mode, bulk_warps=warps, graph_steps=2,
                         prefetch=5 if warps == 8 else 0)
                for n in (1, 4, 3):
                    ens.step(n)
                    ens.sync()
                out += [m.populations() for m in members]
                ens.close()
    return out


def test_checked_paths_are_clean_and_equal(tmp_path):
    from paper_2108_08783_gb300 import build
    lib = build.build(out=str(tmp_path / "liblbm_checked.so"),
                      extra=["-DLBM_CHECKED", "-DLBM_ALTERNATE_BYTES=0"])
    res = str(tmp_path / "out.npz")
    r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT, res],
                       env=dict(os.environ, LBM_LIBRARY=lib), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    got = np.load(res)
    want = run()
    assert len(got.files) == len(want)
    for k, w in enumerate(want):
        np.testing.assert_array_equal(got["arr_%d" % k], w)
