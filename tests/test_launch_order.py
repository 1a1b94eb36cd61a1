"""Order of a kernel's steps around dependent launches, read from the sources (no GPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_19378_b200", "csrc")


def kernels():
    """(file, name, body) of every __global__ function in csrc"""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\([^;{]*\)\s*\{", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield f, m.group(1), src[m.end():i]


def test_tensor_memory_is_taken_between_the_wait_and_the_trigger():
    """Before the wait it could be what the preceding kernel still waits for; after the trigger the following kernel could take
    it first.  Kernels that neither wait nor trigger start alone and end alone."""
    seen = 0
    for f, name, body in kernels():
        alloc = body.find("tmem_alloc(")
        steps = {s: body.find(s + "(") for s in ("pdl_wait", "pdl_trigger", "pdl_join")}
        if alloc < 0 or max(steps.values()) < 0:
            continue
        seen += 1
        assert steps["pdl_join"] < 0, f"{f}: {name} triggers as it waits and takes tensor memory"
        assert 0 <= steps["pdl_wait"] < alloc < steps["pdl_trigger"], f"{f}: {name}"
    assert seen >= 3, seen
