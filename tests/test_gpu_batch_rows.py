"""The batched field step on rows of nodes: instances of even and odd nx, of
four and eight planes per warp and narrower than a warp together in one
launch, against the same batch with its separate Faraday and Ampere phases
(the fluid phase is the same); bit for bit, in two storage forms."""
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402

SHAPES = [(32, 16, 16), (5, 3, 4), (9, 17, 15), (33, 31, 32), (33, 32, 32), (40, 45, 33), (3, 3, 3), (70, 40, 62)]


@pytest.mark.parametrize("storage", [W.F32, W.F16])
def test_batched_rows_equal_separate_phases(storage):
    ws = [W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.3 + 0.1 * i, tau=0.6, z0=0.1 * nz, storage=storage)
          for i, (nz, ny, nx) in enumerate(SHAPES)]
    with lbm.Simulation(ws) as a, lbm.Simulation(ws) as b:
        b.set_field_fusion(lbm.Simulation.FUSION_OFF)
        for n in (5, 4):  # an odd number of steps, then across an export
            a.step(n)
            b.step(n)
            for i in range(len(ws)):
                for x, y in zip(a.get_state(instance=i), b.get_state(instance=i)):
                    assert torch.equal(x, y), (i, SHAPES[i])
