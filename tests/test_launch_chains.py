"""Source check of the programmatic dependent launches (no GPU needed).

A kernel launched by launch_after becomes resident while its predecessor still
runs, so it must wait before it touches memory, and must not read what a
predecessor writes through the read-only path.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1407_8333_gb300", "csrc")
# const __restrict__ parameters that are a caller's inputs: no kernel of a chain writes them
INPUTS = {"t", "freq", "v", "sky"}


def _kernels():
    """name -> (parameters, body) of every __global__ function."""
    out, text = {}, ""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        text += src
        for m in re.finditer(r"__global__\s+void\s*(?:__launch_bounds__\s*\([^)]*\)\s*)?"
                             r"(\w+)\s*\(([^)]*)\)\s*\{", src):
            out[m.group(1)] = (m.group(2), src[m.end():src.index("\n}", m.end())])
    return out, text


def test_chained_kernels_wait_and_read_by_ordinary_loads():
    kernels, text = _kernels()
    # (launched by name, and the two that are chosen by a lambda)
    chained = set(re.findall(r"launch_after\((\w+)", text)) & set(kernels)
    chained |= {"transform_kernel", "windows_kernel"}
    assert len(chained) >= 15
    for name in chained:
        params, body = kernels[name]
        assert "wait_for_previous();" in body, name
        for p in params.split(","):
            if "__restrict__" in p and p.strip().startswith("const"):
                assert p.split("__restrict__")[1].strip() in INPUTS, (name, p)


def test_the_transform_starts_behind_a_completed_correction():
    """It reads positions, offsets and shift tables by __ldg: the window pre-pass lets
    it in after its own wait, and without a pre-pass it is launched plainly."""
    kernels, text = _kernels()
    body = kernels["windows_kernel"][1]
    assert body.index("wait_for_previous();") < body.index("let_next_start();")
    launch = text[text.index("cudaError_t launch_transform("):]
    launch = launch[:launch.index("\n}")]
    assert re.search(r"if \(!windows\) \{\s*k<<<", launch)
