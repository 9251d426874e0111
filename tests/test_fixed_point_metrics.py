"""The fixed-point operator's sources (no GPU)."""
import os
import re

from paper_2005_13425_gb300 import metrics

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_13425_gb300", "csrc")


def included(name, seen):
    if name in seen or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    for inc in re.findall(r'^#include "([^"]+)"', open(os.path.join(CSRC, name)).read(), re.M):
        included(inc, seen)
    return seen


def test_digest_covers_the_head_kernel():
    """A change of any source of the head's kernel outdates its recorded traffic."""
    assert {f for f in included("ax_fx_kernel.cuh", set()) if "/" not in f} - {"internal.cuh"} == set(metrics.CG_HEAD_SOURCES)
