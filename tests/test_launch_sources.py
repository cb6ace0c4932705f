"""Kernels that start before their predecessor has finished (programmatic dependent launch) read what
it wrote: in the CUDA sources every kernel launched that way waits before it touches global
memory, and neither it nor the device code it calls promises the compiler (__restrict__) that data
written by an earlier kernel of the stream does not change during its lifetime."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_04534_gb300", "csrc")
# written before a chain of such launches begins: geometry, inverse diagonal, batch descriptors
FIXED = {"geom", "dinv", "jobs"}


def sources():
    out = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) +
                    glob.glob(os.path.join(CSRC, "*.h"))):
        out[os.path.basename(p)] = re.sub(r"//[^\n]*", "", open(p).read())
    return out


def matching(s, i, a, b):
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == a) - (s[j] == b)
        if depth == 0:
            return j
    raise AssertionError("unbalanced")


def functions(text, qualifier):
    """(name, parameters, body) of the functions with this qualifier"""
    for m in re.finditer(qualifier + r"\b", text):
        head = re.compile(r"(\w+)\s*\(").search
        pos = m.end()
        while True:
            h = head(text, pos)
            end = matching(text, h.end() - 1, "(", ")")
            if h.group(1) != "__launch_bounds__":
                break
            pos = end
        rest = text[end + 1:].lstrip()
        if not rest.startswith("{"):
            continue  # a declaration
        b = text.index("{", end)
        yield h.group(1), text[h.end():end], text[b:matching(text, b, "{", "}") + 1]


def restricted(code):
    return set(re.findall(r"__restrict__\s+(\w+)", code)) - FIXED


def early_kernels():
    found = {}
    for name, text in sources().items():
        for fn, params, body in functions(text, "__global__ void"):
            if "pdl_enter()" in body:
                found[fn] = (name, params, body)
    return found


def test_every_early_launched_kernel_waits_first():
    kernels = early_kernels()
    launched = set()
    for text in sources().values():
        launched |= set(re.findall(r"launch_pdl\(\s*(\w+)\s*<", text))
        for m in re.finditer(r"h\.kernel\s*=\s*([^;]+);", text):  # Shape::kernel, launched by launch_pdl
            launched |= set(re.findall(r"(apply_\w+)<", m.group(1)))
    assert len(launched) >= 12
    for fn in launched:
        assert fn in kernels, f"{fn} is launched early and never waits"
        before = kernels[fn][2].split("pdl_enter()")[0]
        # before the wait: constants, shared memory, its initialisation by thread index
        for line in re.split(r"[;{}]", before):
            line = line.strip()
            assert (not line or line.startswith(("constexpr", "using", "__shared__", "extern __shared__")) or
                    re.fullmatch(r"if \(threadIdx\.x == 0\) jheld = -1", line)), (fn, line)


def test_early_launched_kernels_do_not_restrict_what_earlier_kernels_write():
    kernels = early_kernels()
    assert len(kernels) >= 12
    for fn, (name, params, body) in kernels.items():
        assert not restricted(params) and not restricted(body), (name, fn, restricted(params) | restricted(body))
    for name, text in sources().items():
        for fn, params, body in functions(text, "__device__ __forceinline__ [\\w<>:]+"):
            if fn == "pdl_enter":
                continue
            assert not restricted(params) and not restricted(body), (name, fn, restricted(params) | restricted(body))
    job = re.search(r"struct ApplyJob \{.*?\n\};", sources()["mf_internal.h"], re.S).group(0)
    assert not restricted(job)
