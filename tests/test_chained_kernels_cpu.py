"""Kernels launched with programmatic dependent launch may be resident while
the kernel before them still writes their input, so no source that holds one
reads through the read-only path (__ldg), whose data must not change while a
kernel runs. Read from the sources: launch.cuh's users and what they include."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_05473_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def reached(name, seen):
    if name in seen or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    for inc in re.findall(r'#include "([^"]+)"', code(name)):
        reached(inc, seen)
    return seen


def test_no_read_only_loads_in_chained_kernels():
    users = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and '"launch.cuh"' in code(f)]
    assert {"fluid.cu", "fields.cu", "adjoint.cu", "axi.cu", "aux.cu", "fluid_mom.cu"} <= set(users)
    files = set()
    for u in users:
        reached(u, files)
    bad = [f for f in sorted(files) if "__ldg(" in code(f) or "ld.global.nc" in code(f)]
    assert not bad, bad


def test_chained_kernels_wait_first():
    """Each kernel handed to launch_chained opens with its wait."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu") or "launch_chained(" not in code(f):
            continue
        src = code(f)
        names = set()
        for call in re.findall(r"launch_chained\(([^;]*);", src):
            names |= set(re.findall(r"\b(\w+_kernel)\b", call))
        assert names
        for k in names:
            body = re.search(r"\b%s\([^{]*\)\s*\{\s*(\w+)\(" % k, src)
            assert body and body.group(1) in ("chain_begin", "chain_wait"), (f, k)
