"""Recordings one after another on one handle: the allocations of the one
before are taken over where they fit, and a checkpoint's populations are
written and read in place. Gradients and states equal those of a handle that
records once, for the same, a smaller, a differently cut and a larger
recording, with every state a checkpoint and with steps taken in between."""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("storage", [W.F32, W.F16])
def test_recordings_in_a_row(storage):
    w = W.parity_small().replace(nx=20, ny=13, nz=33, alpha=0.5, z0=2.0, tau=0.6, storage=storage)
    seed = np.random.default_rng(3).standard_normal((3, w.nz, w.ny, w.nx)).astype(np.float32)
    with lbm.Simulation(w) as a:
        for T, K in ((9, 4), (9, 4), (8, 3), (7, 1), (6, 6), (30, 5), (5, 2)):
            a.record(T, K)
            sa = [t.clone() for t in a.get_state()]
            a.step(3)  # the sweep leaves the handle at step T again
            ga = a.adjoint_step(seed)
            for x, y in zip(a.get_state(), sa):
                assert torch.equal(x, y)
            with lbm.Simulation(w) as b:
                b.step(T)
                for x, y in zip(b.get_state(), sa):
                    assert torch.equal(x, y)
                b.record(T, K)
                gb = b.adjoint_step(seed)
            assert np.allclose(ga, gb, rtol=1e-12, atol=0), (T, K, ga, gb)
            ga2 = a.adjoint_step(seed)  # recomputing every segment
            assert np.allclose(ga, ga2, rtol=1e-12, atol=0)
