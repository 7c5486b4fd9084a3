"""Calls made while the caller captures the handle's stream into a graph of
its own. pwfa_lbm_step may be captured: its launches, chained to one another
(programmatic dependent launch), replay as the steps they were, for each form
of the field step. pwfa_lbm_record may not, whether it would allocate or take
over an earlier recording's allocations: it returns PWFA_ERR_CUDA and the
earlier recording stays usable."""
import ctypes
import json
import os
import re
import subprocess
import sys

import pytest

from paper_2201_05473_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2201_05473_gb300 import lbm  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("shape,fusion,boundary", [
    ((64, 32, 32), 1, W.OPEN), ((65, 66, 94), 1, W.OPEN), ((40, 37, 33), 0, W.OPEN),
    ((40, 37, 33), 2, W.PERIODIC), ((64, 32, 32), 1, W.PERIODIC)])
def test_captured_steps_replay(shape, fusion, boundary):
    nz, ny, nx = shape
    w = W.parity_small().replace(nx=nx, ny=ny, nz=nz, alpha=0.5, tau=0.6, z0=2.0, boundary=boundary)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), lbm.Simulation(w, stream=st) as a, lbm.Simulation(w, stream=st) as b:
        for s in (a, b):
            s.set_field_fusion(fusion)
            s.step(3)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            a.step(2)
        g.replay()
        b.step(2)
        st.synchronize()
        for x, y in zip(a.get_state(), b.get_state()):
            assert torch.equal(x, y)


CHILD = r"""
import json, sys
sys.path.insert(0, %(root)r)
import numpy as np, torch
from paper_2201_05473_gb300 import lbm, workloads as W
lbm.load(build=False)
w = W.parity_small().replace(nx=20, ny=13, nz=33, alpha=0.5, z0=2.0, tau=0.6)
seed = np.random.default_rng(3).standard_normal((3, w.nz, w.ny, w.nx)).astype(np.float32)
out = {}
s = torch.cuda.Stream()
with torch.cuda.stream(s):
    sim = lbm.Simulation(w, stream=s)
    if %(recorded)r:
        sim.record(6, 3)
    sim.step(1)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    g.capture_begin(capture_error_mode="thread_local")
    try:
        sim.record(6, 3)
        out["code"] = 0
    except lbm.LBMError as e:
        out["code"], out["msg"] = e.code, str(e)
    try:
        g.capture_end()
    except Exception as e:
        out["capture_end"] = type(e).__name__
    torch.cuda.synchronize()
    try:
        if not %(recorded)r:
            sim.record(6, 3)
        ga = sim.adjoint_step(seed)
        with lbm.Simulation(w, stream=s) as b:
            b.record(6, 3)
            gb = b.adjoint_step(seed)
        out["equal"] = bool(np.allclose(ga, gb, rtol=1e-12, atol=0))
    except lbm.LBMError as e:
        out["after"] = str(e)
    sim.close()
print("RESULT " + json.dumps(out))
"""


@pytest.mark.parametrize("recorded", [False, True])
def test_record_is_refused_under_capture(recorded):
    """In a child process: the refused call invalidates the caller's capture."""
    cp = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT, "recorded": recorded}], capture_output=True,
                        text=True, timeout=300)
    assert cp.returncode == 0, cp.stderr[-3000:]
    r = json.loads([ln for ln in cp.stdout.splitlines() if ln.startswith("RESULT ")][-1][len("RESULT "):])
    assert r["code"] == -2 and "captur" in r["msg"].lower(), r  # PWFA_ERR_CUDA
    assert r.get("equal"), r


def fluid_kernels(sim, stream, path):
    """Names of the fluid kernels that one step launches, from a capture of
    the step."""
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    st, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(st, 1) == 0
    sim.step(1)
    assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) == 0
    assert rt.cudaGraphDebugDotPrint(graph, str(path).encode(), 1) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return set(re.findall(r"fluid_(?:linear_|staged_)?kernel", path.read_text()))


def test_launch_shape_round_trip(tmp_path):
    """What get_launch reports gives another handle the same kernel: the
    default's runs of nodes, and a block shape."""
    w = W.parity_small().replace(nx=131, ny=24, nz=24, storage=W.F16, collision=W.REGULARIZED)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), lbm.Simulation(w, stream=st) as a, lbm.Simulation(w, stream=st) as b:
        for shape, kernel in ((None, "fluid_linear_kernel"), ((32, 4), "fluid_kernel"),
                              ((64, 2), "fluid_linear_kernel")):
            if shape:
                a.set_launch(*shape)
            b.set_launch(*a.get_launch())
            assert b.get_launch() == a.get_launch()
            a.step(2)
            b.step(2)
            st.synchronize()
            for s in (a, b):
                assert fluid_kernels(s, st, tmp_path / "step.dot") == {kernel}
