"""Kernels that start while the launch before them still runs (programmatic dependent launch), checked in
their sources: the populations that such a kernel reads are still being written when its lifetime begins,
so it must not declare them __restrict__ (which promises that nothing else writes what is read through the
pointer while the kernel runs, and allows loads above the wait or through the non-coherent path)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_4736_gb300", "csrc")


def _kernels():
    """(name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        text = re.sub(r"__launch_bounds__(\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\))", "", text)
        for m in re.finditer(r"__global__\s+void\s+(\w+)\(([^{;]*?)\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield m.group(1), m.group(2), text[m.end():end]


def _chained():
    out = [k for k in _kernels() if re.search(r"griddepcontrol|\b(grid_dependency_wait|grid_launch_dependents|batch_begin)\(", k[2])]
    assert {"k_step", "k_step_lanes", "k_step_tma", "k_step_dd", "k_ghost", "k_wall", "k_step_batch"} <= {k[0] for k in out}
    return out


def test_chained_kernels_do_not_promise_that_nobody_writes_their_populations():
    for name, params, _ in _chained():
        assert not re.search(r"\b(R|double|float) \*__restrict__", params), name


def test_chained_kernels_wait_before_anything_else_of_their_grid():
    """A grid reads the results of earlier launches only behind its own griddepcontrol.wait: every kernel that
    is launched so waits, whatever its arguments, and before it reads populations or tables."""
    for name, _, body in _chained():
        at = body.find("grid_dependency_wait();")
        assert at >= 0, name
        before = body[:at]
        assert not re.search(r"\bif\s*\([^)]*$", before), name                    # not conditional
        assert not re.search(r"\b(fin|f|Pall|G|TG|tiles)\s*\[|->|\bload\(|cp\.async", before), name
