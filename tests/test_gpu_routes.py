"""Which launches a call makes, and results that the equality tests between
routes leave open: AUTO takes the fused field step on open grids (counted
launches), the recording's default interval follows the sizes it compares,
and the fused step diagnostics equal a reduction of the state they entered
with, whatever the collision, storage and row length."""
import math

import numpy as np
import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402


def box(shape, **kw):
    nz, ny, nx = shape
    return W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=0.1 * nz, **kw)


@pytest.mark.parametrize("shape,window", [
    ((3, 3, 3), False), ((17, 5, 97), True), ((40, 50, 63), True), ((117, 91, 101), False),  # single nodes
    ((65, 64, 64), True), ((80, 66, 94), False), ((131, 62, 126), True),                     # pairs
])
def test_auto_is_fused_on_open_grids(shape, window):
    """One Faraday launch at the start; with a window, one more before a step
    that moves the box."""
    w = box(shape)
    if window:
        w = w.replace(moving_window=1, window_z=w.z0 + 0.05)
    with lbm.Simulation(w) as s:
        s.step(13)
        _, n = s.kernel_times()
        moves = s.window_planes()
        assert moves == (2 if window else 0)
        assert n["fluid"] == 13 and n["ampere"] == 13 and n["faraday"] == 1 + moves


def test_auto_is_fused_in_a_batch():
    ws = [box(s) for s in ((32, 16, 16), (5, 3, 4), (33, 31, 32))]
    with lbm.Simulation(ws) as s:
        s.step(8)
        _, n = s.kernel_times()
        assert n["faraday"] == len(ws) and n["fluid"] == 8 and n["ampere"] == 8


def align(v):
    return (v + 255) // 256 * 256


def one_segment(w, steps):
    """Whether nsteps as one segment take no more bytes than every
    ceil(sqrt(nsteps)): checkpoints of 76 populations and 6 fields, a segment
    of two population buffers, 6 K + 3 guarded fields and 4 K lattice sums."""
    fb = align((w.nodes + 31) // 32 * 32 * 76 * (4 if w.storage == W.F32 else 2))
    vb = align(4 * w.nodes)
    guarded = vb + align(4 * (w.nx * w.ny + w.nx + 1))
    size = [((steps + k - 1) // k + 1) * (fb + 6 * vb) + 2 * fb + (6 * k + 3) * guarded + 4 * k * vb
            for k in (steps, min(steps, math.ceil(math.sqrt(steps))))]
    return size[0] <= size[1]


@pytest.mark.parametrize("storage,steps,one", [
    (W.F32, 65, True), (W.F32, 66, False), (W.F32, 72, False), (W.F32, 73, True), (W.F32, 74, False),
    (W.F16, 18, True), (W.F16, 19, False), (W.F16, 21, True), (W.F16, 23, False)])
def test_default_interval_follows_the_sizes(storage, steps, one):
    """A sweep over one segment recomputes no step; over checkpoints, all but
    the last segment's."""
    w = box((64, 32, 32), storage=storage)
    assert one_segment(w, steps) == one
    with lbm.Simulation(w) as s:
        s.record(steps)
        s.kernel_times()
        s.adjoint_step()
        _, n = s.kernel_times()
        k = math.ceil(math.sqrt(steps))
        assert n["fluid"] == (0 if one else (math.ceil(steps / k) - 1) * k)


@pytest.mark.parametrize("shape,boundary,collision,storage", [
    ((3, 3, 3), W.OPEN, W.BGK, W.F16), ((5, 7, 11), W.PERIODIC, W.REGULARIZED, W.F32),
    ((8, 4, 128), W.OPEN, W.STREAM_ONLY, W.F32), ((19, 23, 131), W.OPEN, W.REGULARIZED, W.F32),
    ((19, 23, 131), W.OPEN, W.REGULARIZED, W.F16), ((33, 21, 17), W.PERIODIC, W.REGULARIZED, W.BF16),
    ((33, 21, 17), W.OPEN, W.BGK, W.BF16)])
def test_step_diagnostics_against_the_entering_state(shape, boundary, collision, storage):
    """Sums of 19 FP32 values in another order (19 2^-24 = 1.1e-6 of their
    magnitudes), then warp sums of 32 (2e-6): 1e-5 of the sums of magnitudes
    with a margin of three for values that cancel; minimum and maximum 1e-5 of
    themselves; the energy, whose terms are the same, 2e-6."""
    w = box(shape, boundary=boundary, collision=collision, storage=storage)
    with lbm.Simulation(w) as s:
        s.step(6)
        mask = [lbm.FIELD_N, lbm.FIELD_PX, lbm.FIELD_PY, lbm.FIELD_PZ, lbm.FIELD_UX, lbm.FIELD_UY, lbm.FIELD_UZ]
        v = [s.fields(m).cpu().numpy().astype(np.float64).reshape(-1) for m in mask]
        raw = [s.fields(m | lbm.RAW_YEE).cpu().numpy().astype(np.float64)
               for m in (lbm.FIELD_EX, lbm.FIELD_EY, lbm.FIELD_EZ, lbm.FIELD_BX, lbm.FIELD_BY, lbm.FIELD_BZ)]
        d = s.step_diag(1)[0]
        for k in range(4):
            assert abs(d[k] - v[k].sum()) <= 1e-5 * np.abs(v[k]).sum(), k
        energy = 0.5 * w.dx ** 3 * sum((r * r).sum() for r in raw)
        assert abs(d[4] - energy) <= 2e-6 * energy
        assert abs(d[5] - v[0].min()) <= 1e-5 * v[0].max() and d[7] == 0
        top = np.sqrt((v[4] ** 2 + v[5] ** 2 + v[6] ** 2).max())
        assert abs(d[6] - top) <= 1e-5 * top
