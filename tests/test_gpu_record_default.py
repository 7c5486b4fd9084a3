"""The recording's own choice of interval (ckpt_every = 0: checkpoints, or one
segment where that takes no more memory) against stated intervals: the same
states bit for bit, the same gradient up to the order of the FP64 sums; on
both sides of the line, first and second sweep, in FP32 and FP16 storage."""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("storage,steps", [(W.F32, 1), (W.F32, 40), (W.F32, 90), (W.F16, 18), (W.F16, 40)])
def test_default_interval(storage, steps):
    w = W.parity_small().replace(nx=20, ny=13, nz=33, alpha=0.5, z0=2.0, tau=0.6, storage=storage)
    seed = np.random.default_rng(3).standard_normal((3, w.nz, w.ny, w.nx)).astype(np.float32)
    with lbm.Simulation(w) as a, lbm.Simulation(w) as b:
        a.record(steps)
        b.record(steps, int(np.ceil(np.sqrt(steps))))
        for x, y in zip(a.get_state(), b.get_state()):
            assert torch.equal(x, y)
        for _ in range(2):
            ga, gb = a.adjoint_step(seed), b.adjoint_step(seed)
            assert np.all(np.isfinite(ga)) and np.allclose(ga, gb, rtol=1e-12, atol=0), (ga, gb)
        for x, y in zip(a.get_state(), b.get_state()):
            assert torch.equal(x, y)
