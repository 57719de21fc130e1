"""Order of the waits in the conv net's kernels, read from their source.

They are launched while the kernel before them may still run.  A bounded wait whose clock starts before
the wait for that kernel (pdl_wait) counts its run time, and would report a time-out that is not one.
"""
import os
import re

import pytest

import paper_2602_12242_gb300

SRC = os.path.join(os.path.dirname(paper_2602_12242_gb300.__file__), "csrc", "cnn.cu")


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
