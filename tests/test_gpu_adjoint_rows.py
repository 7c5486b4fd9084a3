"""The reverse fluid step on runs of nodes: rows that end at, before and after
a warp's end, rows shorter than a warp (walls of several rows in one warp),
the narrowest grids, both boundaries and collisions. Gradient of a random
functional of E against the oracle's forward-mode derivatives in FP64. Bar:
the relative error 1e-4 of every adjoint test; the FP32 reverse sweep rounds
each step's adjoint at 2^-24, the sums of a few dozen steps stay below 1e-5.
"""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("boundary,collision,shape", [
    (W.OPEN, W.BGK, (31, 9, 12)), (W.OPEN, W.REGULARIZED, (32, 9, 12)), (W.OPEN, W.BGK, (32, 8, 12)),
    (W.OPEN, W.BGK, (33, 9, 12)), (W.OPEN, W.REGULARIZED, (5, 11, 13)), (W.OPEN, W.BGK, (4, 11, 13)),
    (W.OPEN, W.REGULARIZED, (65, 7, 8)), (W.OPEN, W.BGK, (64, 6, 9)),
    (W.PERIODIC, W.BGK, (33, 9, 12)), (W.PERIODIC, W.REGULARIZED, (32, 8, 12))])
def test_gradient_on_ragged_rows(boundary, collision, shape):
    nx, ny, nz = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, boundary=boundary, collision=collision, alpha=0.4,
                                 sigma_r=0.6, sigma_z=0.5, z0=0.8, tau=0.7)
    if boundary == W.OPEN:
        w = w.replace(profile=np.linspace(1.0, 0.7, 8), profile_rmax=1.2)
    steps, np_prof = 24, 8 if boundary == W.OPEN else 0
    rng = np.random.default_rng(nx)
    seed = rng.standard_normal((3, nz, ny, nx))
    d = np.zeros((4 if np_prof else 3, 3 + np_prof))
    d[0, 0] = d[1, 1] = d[2, 2] = 1.0
    if np_prof:
        d[3, 3:] = rng.uniform(0.5, 1.0, np_prof)
    oracle.build()
    _, dE = oracle.tangent_run(steps, d, nx, ny, nz, w.dx, w.dt, w.tau, collision=collision, boundary=boundary,
                               couple=w.couple, n0=w.n0, profile=w.profile, profile_rmax=w.profile_rmax,
                               alpha=w.alpha, sigma_r=w.sigma_r, sigma_z=w.sigma_z, z0=w.z0, n_floor=w.n_floor)
    want = np.array([(seed * e).sum() for e in dE])
    with lbm.Simulation(w) as sim:
        sim.record(steps, 7)
        got = d @ sim.adjoint_step(seed.astype(np.float32))
    # rounding scales with the terms summed, not with a sum that cancels
    scale = np.array([np.sqrt((e ** 2).sum()) for e in dE])
    assert np.all(np.abs(got - want) <= 1e-4 * np.maximum(np.abs(want), scale)), (got, want, scale)
