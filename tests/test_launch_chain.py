"""Sources of the kernels whose launches overlap (csrc/chain.cuh).

Such a kernel runs while the kernel before it still writes.  Data behind a
__restrict__ pointer is promised not to change while the kernel runs, which lets
the compiler load it before the wait at the kernel's start: no pointer of these
kernels, or of a function that they call, may carry the qualifier.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_06798_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _functions(text):
    """name -> (signature, body) of the __global__ and __device__ functions."""
    out = {}
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__(?:global|device)__\b", text):
        brace = text.find("{", m.end())
        semi = text.find(";", m.end())
        if brace < 0 or (0 <= semi < brace):   # a declaration or a variable
            continue
        sig = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", text[m.end():brace])
        name = re.search(r"(\w+)\s*\(", sig)
        if not name:
            continue
        depth, k = 1, brace + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        old = out.get(name.group(1), ("", ""))
        out[name.group(1)] = (old[0] + sig, old[1] + text[brace:k])
    return out


FUNCTIONS = {}
for _f in SOURCES:
    for _n, (_s, _b) in _functions(open(os.path.join(CSRC, _f)).read()).items():
        _o = FUNCTIONS.get(_n, ("", ""))
        FUNCTIONS[_n] = (_o[0] + _s, _o[1] + _b)

CHAINED = sorted(set(re.findall(r"launch_chained\(\s*(\w+)", "".join(open(os.path.join(CSRC, f)).read() for f in SOURCES)))
                 & set(FUNCTIONS))


def _reached(name, seen):
    if name in seen or name not in FUNCTIONS:
        return seen
    seen.add(name)
    for callee in re.findall(r"(\w+)(?:<[^<>;{}]*>)?\s*\(", FUNCTIONS[name][1]):
        _reached(callee, seen)
    return seen


def test_the_chained_kernels_are_found():
    assert {"conv3_kernel", "back3_kernel", "bc_kernel", "step_tile_f32", "tail_kernel"} <= set(CHAINED)


@pytest.mark.parametrize("kernel", CHAINED)
def test_chained_kernels_wait_first_and_promise_no_constant_data(kernel):
    assert re.search(r"chain_begin\(\)|launch_live\(", FUNCTIONS[kernel][1])
    for f in sorted(_reached(kernel, set())):
        assert "__restrict__" not in FUNCTIONS[f][0] + FUNCTIONS[f][1], f


@pytest.mark.parametrize("source,kernel", [("step_f64.cu", "step_tile_f64"), ("step_unsplit.cuh", "step_unsplit_kernel")])
def test_fp64_updates_are_launched_after_their_predecessor(source, kernel):
    """Launched ahead of its end they share SMs unevenly, and each SM's FP64 pipe is what
    bounds them (a 3-level unsplit run took 1.5 times as long).  Only the retake launch,
    which mostly finds nothing to do, overlaps."""
    text = open(os.path.join(CSRC, source)).read()
    plain = text.index("if (a.gate == nullptr) {")
    assert re.match(r"if \(a\.gate == nullptr\) \{\s+" + kernel + r"<[^;]*<<<", text[plain:])
    assert text.index("launch_chained(" + kernel) > plain
