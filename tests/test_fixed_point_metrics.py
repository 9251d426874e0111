"""The fixed-point operator's counts and sources (no GPU)."""
import os
import re

import pytest

from paper_2005_13425_gb300 import metrics

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_13425_gb300", "csrc")


def line_terms(n):
    """Terms of one even-odd line product, counted in the order the kernel forms
    them (fx_line_eo)."""
    h, terms = n // 2, 0
    for _ in range(h):              # the outputs m and n-1-m together
        terms += h + h              # differences and sums
        if n % 2:
            terms += 1              # the middle value
    if n % 2:
        terms += h + 1              # the middle output
    return terms


@pytest.mark.parametrize("n", range(2, 17))
def test_instructions_per_point(n):
    assert metrics.fx_instr_per_point(n) == pytest.approx(3 * (6 * line_terms(n) / n + 9), rel=1e-14)


def test_instructions_at_ten_points():
    assert metrics.fx_instr_per_point(10) == 117
    # three instructions in a group, 33 groups in the time of 121 FFMA
    assert metrics.fx_instr_rate(121.0) == pytest.approx(99.0)


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
