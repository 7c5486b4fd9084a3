"""The steps with separate Faraday and Ampere launches (the PIC driver,
periodic grids, FUSION_OFF, a window's moves): queued back to back, where each
kernel's start overlaps the one before, against the same steps waited for one
at a time. The same kernels on the same data, so the same state bit for bit;
with the PIC driver, whose FP32 atomics add in any order, to 2e-6 of each
array (the rounding of a deposit sum, carried over a few steps)."""
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("kind", ["pic", "periodic", "off", "window"])
@pytest.mark.parametrize("shape,storage,collision", [
    ((33, 21, 19), W.F32, W.BGK), ((64, 32, 32), W.F16, W.REGULARIZED), ((160, 97, 131), W.F32, W.BGK)])
def test_queued_steps_equal_waited_ones(kind, shape, storage, collision):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * nz, storage=storage,
                                 collision=collision)
    if kind == "pic":
        w = w.replace(driver=1)
    if kind == "periodic":
        w = w.replace(boundary=W.PERIODIC)
    if kind == "window":
        w = w.replace(moving_window=1, window_z=w.z0 + 0.05)
    with lbm.Simulation(w) as a, lbm.Simulation(w) as b:
        for s in (a, b):
            if kind == "pic":
                xp, weight = W.bunch_particles(5000, w.alpha, w.sigma_r, w.sigma_z, w.z0, w.dt, w.nx, w.ny, w.dx)
                s.set_particles(xp, weight)
            if kind in ("off", "window"):
                s.set_field_fusion(lbm.Simulation.FUSION_OFF)
        torch.cuda.synchronize()
        a.step(24)
        for _ in range(24):
            b.step(1)
            torch.cuda.synchronize()
        for x, y in zip(a.get_state(), b.get_state()):
            if kind == "pic":
                assert float((x - y).double().norm()) <= 2e-6 * float(y.double().norm())
            else:
                assert torch.equal(x, y)
