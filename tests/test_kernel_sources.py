"""Rules that the kernel sources keep and that no run can show reliably."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1902_01458_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _parameters(src, kernel):
    m = re.search(r"\b%s\s*\(" % kernel, src[src.index("__global__"):])
    start = src.index("__global__") + m.end()
    depth, i = 1, start
    while depth:
        depth += {"(": 1, ")": -1}.get(src[i], 0)
        i += 1
    return [" ".join(p.split()) for p in src[start:i - 1].split(",")]


def test_data_of_a_running_predecessor_is_not_declared_constant():
    """The coupling kernel may start while the product that writes its partial sums
    still runs: const __restrict__ there would promise that they do not change."""
    part = [p for p in _parameters(_source("sweep.cu"), "sweep_couple_kernel")
            if re.search(r"\bpart$", p)]
    assert part == ["const float2* part"]
    rhs = [p for p in _parameters(_source("sweep.cu"), "sweep_tc2_kernel")
           if re.search(r"\brhs$", p)]
    assert rhs == ["const float2* rhs"]


def test_shared_memory_is_opted_in_per_device():
    """The opt-in to more than 48 KB of dynamic shared memory belongs to a device and is
    the same for every call: one helper sets it, and no process-wide flag skips it."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        src = _source(name)
        assert not re.search(r"static\s+(bool|size_t|int)\s+\w*attr", src), name
        calls = src.count("cudaFuncSetAttribute(")
        assert calls == (1 if name == "rr_internal.cuh" else 0), name
