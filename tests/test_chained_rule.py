"""The rule that chained launches rest on, checked in the sources (no GPU): a kernel launched while its predecessor is still
running reads global memory through plain pointers only.  A read-only load (const __restrict__, __ldg, ld.global.nc) is invariant
to the compiler and may be moved above the wait for the predecessor, whatever the wait's "memory" clobber says."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33503_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _functions(src):
    """(name, parameters, body) of every device function and kernel."""
    src = re.sub(r"__(?:launch_bounds|cluster_dims)__\([^()]*\)", "", src)
    for m in re.finditer(r"__(?:global|device)__[^;{}()]*?(?:void|[\w:]+)\s+(\w+)\s*\(", src):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        params, j = src[m.end():i - 1], src.find("{", i)
        if j < 0 or ";" in src[i:j]:
            continue
        k, depth = j + 1, 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            k += 1
        yield m.group(1), params, src[j:k]


def _without_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


@pytest.mark.parametrize("name", [s for s in SOURCES if s.endswith(".cu")])
def test_chained_kernels_read_through_plain_pointers(name):
    src = _without_comments(open(os.path.join(CSRC, name)).read())
    functions = list(_functions(src))
    chained = [f for f in functions if "griddep_wait()" in f[2]]
    for fn, params, body in chained:
        assert not re.search(r"const\s[^,]*\*\s*__restrict__", params), (name, fn)
    if chained:                                          # helpers of such a kernel are inlined into it
        plain = {f[0] for f in functions if f not in chained and re.search(r"\b" + f[0] + r"<<<|\b" + f[0] + r"<[\w, ]+><<<", src)}
        for fn, params, body in functions:
            if fn not in plain:
                assert not re.search(r"const\s[^,]*\*\s*__restrict__", params), (name, fn)
                assert "__ldg" not in body and "ld.global.nc" not in body, (name, fn)


def test_every_chained_launch_names_a_kernel_that_waits():
    text = {s: _without_comments(open(os.path.join(CSRC, s)).read()) for s in SOURCES}
    waits = {f[0] for src in text.values() for f in _functions(src) if "griddep_wait()" in f[2]}
    launched = set()
    for src in text.values():
        for m in re.finditer(r"\blaunch_chained(?:_clusters\(\s*\w+,\s*|\(\s*)(\w+)", src):
            if m.group(1) in ("1", "kernel", "cluster", "void"):
                continue
            alias = re.findall(r"\b" + m.group(1) + r" = (?:[^;]*?\? )?(\w+_kernel)", src[:m.start()])
            launched.add(alias[-1] if alias else m.group(1))
    assert len(launched) >= 20, launched
    assert launched <= waits, launched - waits
