"""Loads of a dependently launched kernel stay behind its wait.

Read from the sources: a load through a __restrict__ pointer may go through the
read-only path and be moved above griddepcontrol.wait, so between pdl_enter()
and the kernel's first branch on the solve's state (`return`) such a pointer is
used only after after_wait().
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_16660_gb300", "csrc")


def _matching(s, i, pair):
    depth = 0
    while True:
        depth += (s[i] == pair[0]) - (s[i] == pair[1])
        if depth == 0:
            return i
        i += 1


def _kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\b", text):
        lb = re.compile(r"\s*__launch_bounds__\(").match(text, m.end())
        at = _matching(text, lb.end() - 1, "()") + 1 if lb else m.end()
        name = re.compile(r"\s*(\w+)\s*\(").match(text, at)
        end = _matching(text, name.end() - 1, "()")
        body = re.compile(r"\s*\{").match(text, end + 1)
        if body:
            yield name[1], text[name.end():end], text[body.end():_matching(text, body.end() - 1, "{}")]


def unfenced(text):
    """(kernel, pointer) of every load that may be moved above the wait."""
    text = re.sub(r"//[^\n]*", "", text)
    out = []
    for name, params, body in _kernels(text):
        if "pdl_enter();" not in body:
            continue
        span = re.split(r"\breturn\b", body.split("pdl_enter();", 1)[1])[0]
        for p in re.findall(r"\*\s*__restrict__\s+(\w+)", params):
            use = re.search(r"(?<![\w.>])%s\s*\[|\bldg\(\s*%s\b|\b__ldg\(\s*%s\b" % (p, p, p), span)
            fence = re.search(r"\b%s = after_wait\(%s\)" % (p, p), span)
            # static data read before the wait as well needs no fence
            static = re.search(r"\b%s\b" % p, body.split("pdl_enter();", 1)[0])
            if use and not static and not (fence and fence.start() < use.start()):
                out.append((name, p))
    return out


def test_a_load_right_after_the_wait_is_found():
    kernel = ("__global__ void __launch_bounds__(64) k(const double *__restrict__ z, double *__restrict__ p) {\n"
              "    pdl_enter();\n    %s p[0] = z[0];\n    if (z[1] > 0) return;\n}\n")
    assert unfenced(kernel % "") == [("k", "z"), ("k", "p")]
    assert unfenced(kernel % "z = after_wait(z); p = after_wait(p);") == []


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_loads_after_the_wait_are_fenced(path):
    with open(path) as f:
        assert unfenced(f.read()) == []
