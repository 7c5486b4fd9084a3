"""The fluid kernels on runs of consecutive nodes (the default) against the
2D block shapes: the same arithmetic per node, so the same state bit for bit,
whatever the row length, with the remainder of the last run, open and
periodic, through the fused diagnostics and the recorded steps."""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("storage", [W.F32, W.BF16, W.F16])
@pytest.mark.parametrize("shape,boundary,collision", [
    ((3, 3, 3), W.OPEN, W.BGK), ((5, 7, 11), W.PERIODIC, W.REGULARIZED), ((8, 4, 128), W.OPEN, W.BGK),
    ((19, 23, 131), W.OPEN, W.REGULARIZED),
])
def test_runs_equal_block_shapes(shape, boundary, collision, storage):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * nz, boundary=boundary,
                                 collision=collision, storage=storage)
    with lbm.Simulation(w) as a, lbm.Simulation(w) as b:
        b.set_launch(32, 4)
        a.step(7)
        b.step(7)
        da, db = a.step_diag(2), b.step_diag(2)
        assert np.array_equal(da, db)
        sa, sb = a.get_state(), b.get_state()
        for x, y in zip(sa, sb):
            assert torch.equal(x, y)
        a.record(9, 4)  # the recorded steps keep their lattice sums as well
        for x, y in zip(a.get_state(), sb):
            assert torch.equal(x, y)
