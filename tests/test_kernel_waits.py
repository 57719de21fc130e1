"""Order of waits and loads in the kernels that are launched while the kernel before them may still run
(pdl_wait), read from their source.

A bounded wait whose clock starts before the wait for that kernel counts its run time, and would report a
time-out that is not one.  A non-coherent load (__ldg, or through a `const __restrict__` parameter) may be
moved above the wait by the compiler, so only what no kernel of the chain writes is read that way.
"""
import glob
import os
import re

import pytest

import paper_2602_12242_gb300

CSRC = os.path.join(os.path.dirname(paper_2602_12242_gb300.__file__), "csrc")
SRC = os.path.join(CSRC, "cnn.cu")

# tables, the tensor, networks' parameters and the forward pass's pre-activations (last written before
# the kernel before) and material maps
CONSTANTS = {"gpre", "twM", "twP", "twH", "twPy", "twL", "tw", "twx", "twy", "twz", "agl", "nhat", "nhk", "n", "t", "Rm", "R",
             "Wl", "wl", "Q1", "q1", "Q2", "q2", "p.bias", "ms_map", "c.ms_map", "c.ku_map", "c.axis_map"}
# (kernels launched after the one before has ended)
ORDINARY = {"yzh_kernel"}


def device_sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def kernels(text):
    """(name, parameters, body) of the kernels of a source."""
    for m in re.finditer(r"__global__ void[^;{]*?\b(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
        if m[1] != "__launch_bounds__":
            yield m[1], m[2], text[m.end():text.index("\n}\n", m.end())]


def roles(kernel):
    """The source before the roles of a kernel part, and each role's."""
    s = open(SRC).read()
    s = s[re.search(r"\b%s\(const" % kernel, s).end():]
    s = s[:s.index("\n}\n")]
    parts = re.split(r"\n  (?:if \(warp == 0\) \{|\} else if \(warp == 1\) \{|\} else \{)\n", s)
    assert len(parts) == 4, len(parts)
    return parts[0], parts[1:]


@pytest.mark.parametrize("kernel", ["conv_tc_kernel", "wgrad_tc_kernel"])
def test_every_role_waits_for_the_kernel_before_first(kernel):
    head, body = roles(kernel)
    for role in body:
        first = re.search(r"(role|mbar)_wait\(", role)
        assert first
        assert "pdl_wait" in head + role[:first.start()]


def test_kernels_that_start_early_take_only_constants_as_const_restrict():
    seen = 0
    for f in device_sources():
        for name, par, body in kernels(open(f).read()):
            if "pdl_wait" not in body:
                continue
            seen += 1
            for p in par.split(","):
                if "const" in p and "__restrict__" in p:
                    assert re.search(r"(\w+)\s*$", p)[1] in CONSTANTS, (os.path.basename(f), name, p.strip())
    assert seen >= 30


def test_non_coherent_loads_read_only_constants():
    for f in device_sources():
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for name, _, body in kernels(text):
            if name in ORDINARY:
                text = text.replace(body, "")
        for m in re.finditer(r"(?:__ldg|ldg4)\((?:reinterpret_cast<const float[24]\*>\()?&?([\w.]+)", text):
            if m[1] in ("const", "p") or "ldg4(a +" in text[m.start():m.end() + 3]:
                continue  # (ldg4's own definition, load3<FAR>'s; twiddle rows)
            assert m[1] in CONSTANTS, (os.path.basename(f), m[1], text[m.start():m.end() + 20])
