"""Rules of the kernel sources that no run can show reliably (a violation is a fault or a race that depends on timing), read off
the text of csrc/ and of the probe kernels."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05838_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
PROBES = sorted(glob.glob(os.path.join(os.path.dirname(os.path.abspath(__file__)), "probe", "*.cu")))


def code_lines(path):
    """(line number, text) without // comments."""
    with open(path) as f:
        return [(i + 1, re.sub(r"//.*", "", line)) for i, line in enumerate(f)]


def unsynced_tensor_memory_access(lines):
    """Line numbers of warp-collective tensor-memory instructions that follow a polling wait, or (deallocation) anything at
    all, without a __syncwarp() or warp vote between: the lanes of a warp may arrive there one by one."""
    bad, split = [], False
    for i, (no, text) in enumerate(lines):
        if re.search(r"\bMDN_(WAIT|SPIN)\(b|\bmbar_wait(_spin)?\(", text):
            split = True
        if re.search(r"__global__|__syncwarp\(|__all_sync\(|\bwait_all\(", text):
            split = False
        if re.search(r"\b(tmem_(ld|st)(16|32|_n)|load16)\b[<(]", text) and split and "__device__" not in text:
            bad.append(no)
        if "tmem_dealloc(" in text and not any("__syncwarp()" in t for _, t in lines[max(0, i - 3):i]):
            bad.append(no)
    return bad


@pytest.mark.parametrize("path", [p for p in SOURCES + PROBES if "tmem_dealloc(" in open(p).read()], ids=os.path.basename)
def test_warps_reconverge_before_tensor_memory_instructions(path):
    assert unsynced_tensor_memory_access(code_lines(path)) == []


def kernels(lines):
    """The lines of every __global__ function: (name, lines)."""
    out = []
    for no, text in lines:
        if "__global__" in text:
            out.append([None, []])
        if out:
            out[-1][1].append((no, text))
            m = re.search(r"\b(\w+_kernel)\(", text)
            if out[-1][0] is None and m:
                out[-1][0] = m.group(1)
    return out


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_kernel_lets_its_dependents_in_before_its_own_wait(path):
    """Kernels that are let in early read the call's inputs before their wait: that needs every kernel in front of them to
    have waited for its own predecessor first."""
    for name, lines in kernels(code_lines(path)):
        calls = [(m.group(0), no) for no, t in lines for m in re.finditer(r"grid_(dependency_wait|launch_dependents)(?=\(\))", t)]
        if any(c == "grid_launch_dependents" for c, _ in calls):
            assert calls[0][0] == "grid_dependency_wait", (name, calls)
