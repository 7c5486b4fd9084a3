"""The diagnostics of a state against FP64 reductions of its exported node
fields (the same FP32 moments): sums to the rounding of FP64 sums (N 2^-53 of
the sum of magnitudes, below 1e-12 at these sizes), minimum, count and maximum
|beta| exactly (one FP64 root); sizes below one run of nodes, with a ragged
last run and with several runs per block, all storage forms, both boundaries,
at rest and driven. And the step's own diagnostics, whose warps sum in FP32
(32 values: 2e-6), against those of the state it entered with."""
import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("shape,storage,boundary,steps", [
    ((3, 3, 3), W.F32, W.OPEN, 2), ((7, 6, 6), W.F16, W.PERIODIC, 3), ((33, 21, 17), W.BF16, W.OPEN, 6),
    ((40, 33, 31), W.F32, W.PERIODIC, 6), ((129, 65, 67), W.F32, W.OPEN, 9), ((129, 65, 67), W.F16, W.OPEN, 0)])
def test_diagnostics_against_fields(shape, storage, boundary, steps):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * nz, storage=storage,
                                 boundary=boundary)
    with lbm.Simulation(w) as sim:
        if steps:
            sim.step(steps)
        names = [lbm.FIELD_N, lbm.FIELD_PX, lbm.FIELD_PY, lbm.FIELD_PZ, lbm.FIELD_UX, lbm.FIELD_UY, lbm.FIELD_UZ]
        n, p0, p1, p2, u0, u1, u2 = [sim.fields(m).cpu().numpy().astype(np.float64).reshape(-1) for m in names]
        raw = [sim.fields(m | lbm.RAW_YEE).cpu().numpy().astype(np.float64).reshape(-1)
               for m in (lbm.FIELD_EX, lbm.FIELD_EY, lbm.FIELD_EZ, lbm.FIELD_BX, lbm.FIELD_BY, lbm.FIELD_BZ)]
        d = sim.diag()
        energy = 0.5 * w.dx ** 3 * sum((r * r).sum() for r in raw)
        for got, v in zip(d[:4], (n, p0, p1, p2)):
            assert abs(got - v.sum()) <= 1e-12 * np.abs(v).sum()
        assert abs(d[4] - energy) <= 1e-12 * energy
        assert d[5] == n.min() and d[7] == 0
        assert abs(d[6] - np.sqrt((u0 * u0 + u1 * u1 + u2 * u2).max())) <= 4e-16 * d[6]
        out = np.empty((1, 8))
        sim.step_diag(1, out=out)
        scale = np.array([np.abs(v).sum() for v in (n, p0, p1, p2)])
        assert np.all(np.abs(out[0, :4] - d[:4]) <= 2e-6 * scale)
        assert abs(out[0, 4] - d[4]) <= 2e-6 * d[4] and out[0, 5] == d[5] and out[0, 7] == 0
        assert abs(out[0, 6] - d[6]) <= 1e-6 * d[6]
