"""Kernels launched with launch_dep may start while the kernel before them still writes.  What that one writes
is not read-only for their life, so a parameter through which a kernel (or a function that it calls) reads
it is not declared `const ... __restrict__`: that would allow the compiler the read-only path.  Checked
in the sources: only what bind writes is so declared."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_08024_gb300", "csrc")

BOUND = {"rowptr", "col", "A", "Dinv", "L", "childptr", "parent", "crow_seg", "crow_off", "cinv_off", "Ainv", "seg_dof",
         "perm0"}


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))}


def parameters(text, name):
    """Parameter lists of the definitions of a function (its name followed by a list and a body)."""
    for m in re.finditer(r"\b%s\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if text[i:].lstrip().startswith("{"):
            yield text[m.end():i - 1]


def test_read_only_parameters_are_what_bind_writes():
    src = sources()
    everything = "\n".join(src.values())
    kernels = set(re.findall(r"launch_dep\((?:flexible \? )?(\w+)", everything)) - {"void"}
    assert {"cg_update_kernel", "bsr_kernel", "fx_kernel", "coarse_kernel", "permute_kernel"} <= kernels
    found = 0
    for name in sorted(kernels | {"partials_sum", "row_acc", "split_row_acc", "split_restrict"}):
        for text in src.values():
            for params in parameters(text, name):
                found += 1
                held = re.findall(r"const [\w ]+\* __restrict__ (\w+)", params)
                assert set(held) <= BOUND, (name, set(held) - BOUND)
    assert found >= len(kernels)
