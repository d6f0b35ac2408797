"""The kernels that run chained (programmatic dependent launch) start while the
kernel before them still writes their inputs.  A pointer marked __restrict__
lets the compiler load through the read-only path, or ahead of the wait, so
those kernels, and the device functions that they call, carry none, and wait
before anything else touches global memory.  Source checks, no GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_23158_gb300", "csrc")
FILES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
         for p in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}


def _functions(text):
    """name -> (signature, body) of the __global__ and __device__ functions."""
    out = {}
    for m in re.finditer(r"__(?:global|device)__[^;{}()]*?(?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        sig = text[m.end():i - 1]
        rest = re.match(r"[\s\w]*\{", text[i:])
        if not rest:
            continue
        j = k = i + rest.end()
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out.setdefault(m.group(1), []).append((sig, text[k:j - 1]))
    return out


FUNCS = {}
for _t in FILES.values():
    for _n, _v in _functions(_t).items():
        FUNCS.setdefault(_n, []).extend(_v)
CHAINED = sorted({m for t in FILES.values() for m in re.findall(r"launch_chained\(\s*chained,\s*(\w+)", t)})


def test_the_chained_kernels_are_found():
    assert {"project_kernel", "onesweep_pass", "emit_fused_kernel", "emit_count_kernel", "emit_scan_kernel",
            "emit_write_kernel", "blend_kernel"} <= set(CHAINED)


@pytest.mark.parametrize("kernel", CHAINED)
def test_inputs_of_chained_kernels(kernel):
    todo, seen = [kernel], set()
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        for sig, body in FUNCS[name]:
            assert "__restrict__" not in sig and "__restrict__" not in body, name
            todo += [c for c in set(re.findall(r"(\w+)\s*(?:<[^;{}()]*>)?\s*\(", body)) if c in FUNCS]


@pytest.mark.parametrize("kernel", CHAINED)
def test_chained_kernels_wait_first(kernel):
    for sig, body in FUNCS[kernel]:
        assert body.count("chain_wait()") == 1
        before = body[:body.index("chain_wait()")]
        pointers = re.findall(r"\*\s*(\w+)\s*(?:,|$)", sig)
        assert not any(re.search(rf"\b{p}\b", before) for p in pointers), kernel
