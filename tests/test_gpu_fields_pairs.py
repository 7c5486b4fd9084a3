"""The fused field step with two nodes per thread (open grids of an even nx)
against the separate Faraday and Ampere kernels: the same arithmetic, so the
same state bit for bit; at each number of planes per warp, at rows shorter
than a warp's nodes and at the line to single nodes, with a moving window."""
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("shape,window", [
    ((65, 64, 62), False), ((65, 64, 64), True),          # below and above the line; two planes
    ((35000, 3, 4), False), ((4097, 32, 2 * 3), False),   # rows shorter than a warp's nodes
    ((200, 3, 450), False), ((3, 300, 300), True),        # one plane per warp
    ((80, 66, 94), False), ((131, 62, 126), True),        # three and four planes
    ((65, 404, 322), False),                              # eight planes
])
def test_pairs_equal_separate_kernels(shape, window):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * min(nz, 130))
    if window:
        w = w.replace(moving_window=1, window_z=w.z0 + 0.05)
    with lbm.Simulation(w) as a, lbm.Simulation(w) as b:
        b.set_field_fusion(lbm.Simulation.FUSION_OFF)
        for n in (9, 4):
            a.step(n)
            b.step(n)
            for x, y in zip(a.get_state(), b.get_state()):
                assert torch.equal(x, y)
