"""A refused cooperative launch: a small lattice goes on with the launched kernels.

The refusal is an error code from a fake of cudaLaunchCooperativeKernel, compiled
into a build of its own (a forced include) that runs in a subprocess: after
`LBM_TEST_LAUNCHES` real launches it returns cudaErrorCooperativeLaunchTooLarge.
The populations equal those of the package's build bit for bit, also when the
refusal comes after the first 1,000 steps of a call.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = r"""
#include <cstdlib>
#include <cuda_runtime.h>
static inline cudaError_t refused(const void* f, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
  static int left = std::atoi(std::getenv("LBM_TEST_LAUNCHES"));
  if (left-- > 0) return cudaLaunchCooperativeKernel(f, g, b, a, m, s);
  return cudaErrorCooperativeLaunchTooLarge;
}
#define cudaLaunchCooperativeKernel refused
"""
SCRIPT = r"""
import sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np
from test_gpu_small_refused import run
np.savez(sys.argv[2], *run())
"""


def run():
    from paper_2108_08783_gb300 import Lattice
    out = []
    for storage in ("f32", "f64", "f16s"):
        geo = I.tube(5, 40, u_mean=0.01, u_amp=0.01, period=37.0)
        lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=0.75)
        lat.set_wall("elastic", rho0=1.0, F=0.85, kappa=6.0)
        for n in (1, 2045, 7):
            lat.step(n)
        lat.sync()
        assert lat.step_count == 2053
        out += [lat.populations(), *lat.wall_state()]
        lat.close()
    return out


def test_refused_launch_falls_back(tmp_path):
    from paper_2108_08783_gb300 import build
    fake = tmp_path / "fake.h"
    fake.write_text(FAKE)
    lib = build.build(out=str(tmp_path / "liblbm_refused.so"), extra=["-include", str(fake)])
    want = run()
    for launches in (0, 2):
        env = dict(os.environ, LBM_LIBRARY=lib, LBM_TEST_LAUNCHES=str(launches))
        res = str(tmp_path / ("out%d.npz" % launches))
        r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT, res], env=env,
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
        got = np.load(res)
        for k, w in enumerate(want):
            np.testing.assert_array_equal(got["arr_%d" % k], w)
