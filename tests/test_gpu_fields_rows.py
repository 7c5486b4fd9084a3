"""The fused field step over rows of nodes (open grids) against the separate
Faraday and Ampere kernels: the same arithmetic, so the same state bit for
bit, at the smallest grids, at odd sizes on both sides of the lines between
its forms, and with a moving window."""
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("shape,window", [
    ((3, 3, 3), False), ((4, 3, 31), False), ((9, 33, 62), False), ((17, 5, 97), True),  # one plane per warp
    ((47, 47, 47), False), ((40, 50, 63), True),                                      # two planes
    ((117, 91, 101), False),                                                          # four planes
])
def test_rows_equal_separate_kernels(shape, window):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * nz)
    if window:
        w = w.replace(moving_window=1, window_z=w.z0 + 0.05)
    with lbm.Simulation(w) as a, lbm.Simulation(w) as b:
        b.set_field_fusion(lbm.Simulation.FUSION_OFF)
        for n in (9, 4):  # 13 steps, two window moves; across an export
            a.step(n)
            b.step(n)
            assert a.window_planes() == b.window_planes()
            for x, y in zip(a.get_state(), b.get_state()):
                assert torch.equal(x, y)
        assert not window or a.window_planes() == 2
