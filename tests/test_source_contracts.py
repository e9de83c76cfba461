"""Contracts of PTX instructions that the compiler does not check and a run seldom
shows broken, checked in the sources of the kernels (no GPU needed)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2405_18628_gb300", "csrc")


def _sources():
    """The CUDA sources by file name, comments taken out."""
    out = {}
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            src = f.read()
        out[name] = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", src, flags=re.S))
    return out


def _bodies(src):
    """Bodies of the device functions of ppd_device.cuh by name (overloads one after the
    other)."""
    out = {}
    for m in re.finditer(r"^PPD_DEV \w[\w ]* (\w+)\(.*?^\}$", src, flags=re.S | re.M):
        out[m.group(1)] = out.get(m.group(1), "") + m.group(0)
    return out


def test_cluster_barriers_are_reached_by_converged_warps():
    """barrier.cluster.*.aligned wants all lanes of a warp at once: every such barrier
    sits behind a __syncwarp() in the one function that issues it, whatever branches its
    callers come from."""
    src = _sources()
    for name, text in src.items():
        if name != "ppd_device.cuh":
            assert "barrier.cluster" not in text, name
    bodies = {f: b for f, b in _bodies(src["ppd_device.cuh"]).items() if "barrier.cluster" in b}
    assert set(bodies) == {"cluster_sync", "cluster_sync_exit"}
    for f, body in bodies.items():
        assert 0 <= body.find("__syncwarp()") < body.find("asm"), f


def test_tensor_memory_loads_are_waited_for_by_name():
    """tcgen05.ld fills its registers some time after it issues, and arithmetic on them
    is free to move across a wait that does not mention them: every wait names the
    registers (in-out operands), and the waits are issued by those functions only."""
    src = _sources()
    for name, text in src.items():
        if name != "ppd_device.cuh":
            assert "wait::ld" not in text, name
    bodies = {f: b for f, b in _bodies(src["ppd_device.cuh"]).items() if "wait::ld" in b}
    assert bodies
    for f, body in bodies.items():
        for stmt in re.findall(r"asm volatile\(\s*\"tcgen05\.wait::ld.*?;\n", body, flags=re.S):
            outs = len(re.findall(r'"\+r"', stmt))
            n = int(re.search(r"\(&r\)\[(\d+)\]", body[:body.index(stmt)].rsplit("PPD_DEV", 1)[1]).group(1))
            assert outs == n, (f, outs, n)


def test_no_load_assumes_that_its_data_never_changes():
    """A grid of a programmatic chain is on the chip while the grids before it still
    write its inputs; it waits for them and then reads.  ld.global.nc (__ldg, or a plain
    load through a const __restrict__ pointer) wants data that stays unchanged for as long
    as the grid exists, so no kernel uses it."""
    for name, text in _sources().items():
        for word in ("__ldg", "global.nc", "__restrict__"):
            assert word not in text, (name, word)
