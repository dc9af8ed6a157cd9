"""Kernels launched as dependent launches start while the kernel before them may still write what they
read.  Their sources therefore declare no pointer __restrict__ (the compiler could then move a load above
the wait, or make it a read-only one) and contain no read-only load."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_04971_gb300", "csrc")
SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
           for p in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}


def _functions(text):
    """(name, signature, body) of every __global__ or __device__ function."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?\b(\w+)\s*\(", text):
        i, depth = text.find("{", m.end()), 0
        if ";" in text[m.end():i]:
            continue
        for j in range(i, len(text)):
            depth += (text[j] == "{") - (text[j] == "}")
            if depth == 0:
                break
        name = re.findall(r"(\w+)\s*\(", text[m.start():i])
        name = next(n for n in name if n not in ("__launch_bounds__", "__align__"))
        yield name, text[m.start():i], text[i:j + 1]


def _dependent_kernels():
    """Signatures of the kernels that wait for the kernel before them, themselves or in a helper."""
    found = {}
    for text in SOURCES.values():
        functions = list(_functions(text))
        waits = {"grid_dependency_wait"} | {n for n, _, body in functions if "grid_dependency_wait()" in body}
        for name, sig, body in functions:
            if "__global__" in sig and any(re.search(rf"\b{w}\s*\(", body) for w in waits):
                found[name] = sig
    return found


def test_dependent_kernels_declare_no_pointer_unaliased():
    kernels = _dependent_kernels()
    launched = {k for text in SOURCES.values() for k in re.findall(r"launch_dependent\((\w+)", text)} - {"void"}
    assert launched and launched | {"score_kernel"} <= set(kernels), launched - set(kernels)
    bad = [k for k, sig in kernels.items() if "__restrict__" in sig]
    assert not bad, bad


def test_no_read_only_loads_beside_dependent_kernels():
    bad = [f for f, text in SOURCES.items() if re.search(r"ld\.global(\.\w+)*\.nc\b|\b__ldg\s*\(", text)
           and ("grid_dependency_wait" in text or f.endswith(".cuh"))]
    assert not bad, bad
