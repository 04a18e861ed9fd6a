"""No kernel lets its successor in before its own blocks end: blocks that come in while some SMs are still taken
are stacked on the others (an FP64 tempering update of 1000 particles on 1/8 took twice as long that way). And every
kernel launched so that it may overlap its predecessor waits for it: launch_after and overlap_attr go with kernels
that call grid_wait()."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_09763_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_successors_come_in_as_blocks_end():
    for path in glob.glob(os.path.join(CSRC, "*")):
        if path.endswith((".cu", ".h", ".cpp")):
            assert "launch_dependents" not in _code(path), path


def test_overlapped_kernels_wait():
    launched = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = _code(path)
        names = set(re.findall(r"launch_after\(\s*(?:[^,?]*\?\s*)?(\w+_kernel)\b", text))
        names |= set(re.findall(r"auto kern = (\w+_kernel\w*)", text)) if "launch_after(kern" in text else set()
        if "overlap_attr(attr" in text:
            names |= set(re.findall(r"cudaLaunchKernelEx\(&cfg, (\w+_kernel)<", text))
        for name in names:
            body = re.search(r"\b%s\((?:[^{;]|\n)*?\)\s*\{(.*?)\n\}" % name, text, re.S)
            assert body and "grid_wait();" in body.group(1), (path, name)
            launched += 1
    assert launched >= 10
