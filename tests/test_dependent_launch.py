"""Kernels that start before their predecessor has finished (csrc/mg_launch.cuh) read its
results in an order that the sources guarantee: by plain loads through pointers without
__restrict__, which the wait's memory clobber orders.  Checked on the sources, on the CPU.
"""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1103_6031_gb300", "csrc")


def sources():
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        with open(path) as f:
            out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", f.read())
    return out


def closing(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise ValueError("unbalanced")


def functions(text, start):
    """(name, parameters, body) of every function whose definition begins with start."""
    for m in re.finditer(start, text):
        n = re.compile(r"\b(k_\w+)\s*\(").search(text, m.end())
        end = closing(text, n.end() - 1, "()")
        brace = text.index("{", end)
        if text[end + 1:brace].strip():
            continue  # a declaration
        yield n.group(1), text[n.end():end], text[brace:closing(text, brace, "{}") + 1]


def test_dependent_kernels_read_by_plain_loads():
    seen = set()
    for name, text in sources().items():
        for kernel, params, body in functions(text, r"__global__"):
            if "grid_wait()" not in body and "_tile<" not in body:
                continue
            seen.add(kernel)
            for p in params.split(","):
                assert not re.search(r"\bconst\b.*\*.*__restrict__", p), (name, kernel, p.strip())
            assert "__ldg(" not in body, (name, kernel)
    launched = set(re.findall(r"launch_dep\(\s*(k_\w+)", " ".join(sources().values())))
    assert len(launched) > 20 and launched <= seen, launched - seen


def test_shared_device_code_reads_by_plain_loads():
    for name in ("mg_stencil.cuh", "mg_tile.cuh", "mg_vbody.cuh", "mg_fixed.cuh", "mg_ghost.cu",
                 "mg_smooth.cu"):
        # the coarsest level's kernel table is written when the hierarchy is made
        left = [a for a in re.findall(r"__ldg\(\s*(\w+)", sources()[name]) if a != "kern"]
        assert not left, (name, left)
