"""The axisymmetric step on runs of consecutive nodes: rows shorter and longer
than a run, a remainder in the last one, every output against the FP64 oracle
(the repository's FP32 bar, 1e-5 of the largest magnitude of each output, over
20 steps from a source with waves), and the chunked source back and forth."""
import numpy as np
import pytest

import oracle
from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("shape", [(5, 5), (3, 200), (64, 4), (9, 127), (8, 128), (7, 129), (130, 31)])
def test_runs_match_oracle(shape):
    nz, nr = shape
    w = W.axisymmetric_parity().replace(nz=nz, nr=nr, tau=0.6, z0=0.1 * nz, alpha=0.5)
    w9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    rng = np.random.default_rng(1)
    A = np.stack([1.0 + 0.1 * rng.standard_normal((nz, nr)), 0.05 * rng.standard_normal((nz, nr)),
                  0.05 * rng.standard_normal((nz, nr))])
    S = (w9[None, :, None, None] * A[:, None]).astype(np.float32)
    refl = [0, 1, 2, 4, 3, 7, 8, 5, 6]
    for q in range(9):
        S[:2, refl[q], :, 0] = S[:2, q, :, 1]
        S[2, refl[q], :, 0] = -S[2, q, :, 1]
    oracle.build()
    o = oracle.AxiOracle(nz, nr, w.dx, w.dt, w.tau, alpha=w.alpha, sigma_r=w.sigma_r, sigma_z=w.sigma_z, z0=w.z0)
    o.set_source(S)
    o.step(20)
    with lbm.AxiSimulation(w) as sim:
        sim.set_source(S)
        assert np.array_equal(sim.get_source().cpu().numpy(), S)
        sim.step(20)
        g = sim.fields().cpu().numpy().astype(np.float64)
    m = o.moments()
    for a, b in zip(g, (m["n"], m["beta_z"], m["beta_r"], *o.get_fields())):
        assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
