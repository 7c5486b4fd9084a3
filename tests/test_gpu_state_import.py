"""The state import (inverse of the pull) and export on odd sizes: distinct
integers come back at every interior node (every node of a periodic grid)
bit for bit in FP32; the 16-bit forms return the one rounding of the stored
deviation."""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("boundary", [W.OPEN, W.PERIODIC])
@pytest.mark.parametrize("shape", [(3, 3, 3), (4, 5, 131), (9, 8, 16), (7, 33, 31)])
def test_integers_come_back(shape, boundary):
    nz, ny, nx = shape
    f = W.integer_populations(shape).astype(np.float32)
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, boundary=boundary)
    with lbm.Simulation(w) as sim:
        sim.set_state(f=f)
        g = sim.get_state(device=False)[0].numpy()
    inner = (slice(None), slice(None)) + (slice(1, -1),) * 3 if boundary == W.OPEN else ()
    assert np.array_equal(g[inner], f[inner])


@pytest.mark.parametrize("storage,u", [(W.BF16, 2.0 ** -8), (W.F16, 2.0 ** -11)])
def test_one_rounding_in_16_bits(storage, u):
    shape = (6, 7, 37)
    f = W.random_populations(shape, seed=5).astype(np.float32)
    w = W.parity_small().replace(nx=37, ny=7, nz=6, boundary=W.PERIODIC, storage=storage)
    wq = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    base = np.zeros((4, 19))
    base[0] = wq
    with lbm.Simulation(w) as sim:
        sim.set_state(f=f)
        g = sim.get_state(device=False)[0].numpy().astype(np.float64)
    dev = np.abs(f - base[:, :, None, None, None])
    # half a unit in the last place of the deviation, and the FP32 roundings
    # of forming it and of adding the base again
    assert np.all(np.abs(g - f) <= 0.5 * 2.0 * u * dev + 2.0 ** -22)
