"""Kernels are launched before the one in front of them has completed, so each has to
wait for it (grid_wait) before it touches memory: as its first statement, or, in
the two training kernels, after reading what no training kernel writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_02840_gb300", "csrc")
LATER = {"k_mlp_grad", "k_adam"}


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", src):
            depth, k = 0, m.end()
            while depth or src[k] not in "{;":
                depth += {"(": 1, ")": -1}.get(src[k], 0)
                k += 1
            if src[k] == "{":
                end = src.find("\n}", k)
                yield re.search(r"\b(k_\w+)\s*\(", src[m.end():k]).group(1), src[k + 1:end]


def test_every_kernel_waits_for_the_one_before():
    found = list(kernels())
    assert len(found) > 80
    for name, body in found:
        if name in LATER:
            assert "grid_wait();" in body, name
        else:
            assert body.lstrip().startswith("grid_wait();"), name


def test_no_launch_goes_round_the_rule():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        assert "<<<" not in re.sub(r"//[^\n]*", "", open(path).read()), path


def test_no_zeros_or_copies_go_unchecked():
    """zero_async and copy_async return their launch's error: each call passes it on."""
    calls = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\b(zero|copy)_async\(", src):
            line = src[src.rfind("\n", 0, m.start()) + 1:m.start()]
            if line.strip() == "int":   # declarations, definitions
                continue
            calls += 1
            assert line.endswith(("CRK_TRY(", "rc = ")), (path, src[m.start() - 40:m.start() + 40])
    assert calls > 30
