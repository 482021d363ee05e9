"""Register budget of the dataflow kernels (heom_flow.cuh), as nvcc reports it: the blocked state array must not cost
them registers in the step loop.  The bounds are what the compiler (CUDA 13.0) gave these kernels when the state was
element-major and a node's own words were at the addresses of its state; keeping both addresses alive took eight sites
with complex H in FP64 from 440 to 1404 bytes of spill stores, at 80 registers a thread instead of 168."""
import os
import re
import subprocess

import pytest

from paper_1012_4382_gb300 import build as heom_build

# (N, complex H, nodes per thread) -> most spill stores and loads (bytes per thread)
FP64 = {(5, True, 1): (144, 144), (6, True, 1): (248, 252), (7, False, 1): (72, 64), (7, True, 1): (1220, 1256),
        (7, False, 2): (0, 0), (8, False, 1): (120, 112), (8, True, 1): (440, 448), (8, False, 2): (4, 12)}
MIXED = {(7, False, 1): (0, 0), (7, True, 1): (40, 32), (8, True, 1): (108, 104)}
FULL_BUDGET = {("double", 8, True, 1)}  # at one CTA's whole register budget, not half of it


@pytest.mark.parametrize("real,limits", [("double", FP64), ("float", MIXED)])
def test_dataflow_kernels_spill_no_more_than_with_an_element_major_state(tmp_path, real, limits):
    src = tmp_path / "flow.cu"
    mixed = "true" if real == "float" else "false"
    src.write_text('#include "heom_flow.cuh"\nnamespace heom { const void* kernels[] = {%s}; }\n' % ", ".join(
        "(const void*)heom_flow_kernel<%d, %s, %s, %s, %d>" % (N, real, mixed, str(c).lower(), npt)
        for N, c, npt in limits))
    r = subprocess.run([heom_build._nvcc()] + heom_build.ARCH + ["-O3", "-std=c++17", "-I" + heom_build.INCLUDE,
                       "-I" + heom_build.CSRC, "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "flow.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    seen = {}
    key = None
    for line in r.stderr.splitlines():
        m = re.search(r"heom_flow_kernelILi(\d)E[df]Lb[01]ELb([01])ELi(\d)E", line)
        if m:
            key = (int(m.group(1)), m.group(2) == "1", int(m.group(3)))
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m:
            spill = (int(m.group(1)), int(m.group(2)))
        m = re.search(r"Used (\d+) registers", line)
        if m:
            seen[key] = spill + (int(m.group(1)),)
    assert set(seen) == set(limits)
    for k, (st, ld) in limits.items():
        assert seen[k][0] <= st and seen[k][1] <= ld, (k, seen[k])
        if (real,) + k in FULL_BUDGET:
            assert seen[k][2] > 84, (k, seen[k])


def test_shared_memory_kernels_keep_their_registers(tmp_path):
    """The kernels of launch mode 2, three and six sites: what the compiler gave their step loops before the state was
    blocked; fewer went with longer steps (the loads of a stage are issued in smaller groups)."""
    src = tmp_path / "smem.cu"
    want = {(3, True): 110, (6, True): 128}
    src.write_text('#include "heom_engine.cuh"\nnamespace heom { const void* kernels[] = {%s}; }\n' % ", ".join(
        "(const void*)heom_smem_kernel<%d, false, %s>" % (N, str(reg).lower()) for N, reg in want))
    r = subprocess.run([heom_build._nvcc()] + heom_build.ARCH + ["-O3", "-std=c++17", "-I" + heom_build.INCLUDE,
                       "-I" + heom_build.CSRC, "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "smem.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    key, seen = None, {}
    for line in r.stderr.splitlines():
        m = re.search(r"heom_smem_kernelILi(\d)ELb0ELb([01])E", line)
        if m:
            key = (int(m.group(1)), m.group(2) == "1")
        m = re.search(r"Used (\d+) registers", line)
        if m:
            seen[key] = int(m.group(1))
    assert seen == want
