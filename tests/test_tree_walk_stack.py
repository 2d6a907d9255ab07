"""The node stack of the group walks (csrc/dwg_tree.cu, grp_walk): a step pops
up to 32 W nodes and pushes the children of the open ones.  The stack stays
sorted by depth, so it never holds more than 32 W (levels + 1) entries, which
is below its W * kGrpStack for any cloud the library takes: no walk of either
pass gives up, whatever opens (CPU model of the walk)."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2405_13839_gb300", "csrc", "dwg_tree.cu")


def _constant(name):
    return int(re.search(rf"constexpr int {name} = (\d+);", open(SRC).read()).group(1))


def _peak(levels, width, open_at, steps=3000):
    stack, peak = [0], 1
    while stack and steps:
        steps -= 1
        pop = stack[-32 * width:]
        del stack[-32 * width:]
        for d in pop:
            if d < levels and open_at(d):
                stack += [d + 1, d + 1]
        peak = max(peak, len(stack))
    return peak


@pytest.mark.parametrize("width", [1, _constant("kWalkW")])
def test_stack_bound(width):
    levels = 27  # 2^31 points in leaves of 16
    bound = 32 * width * (levels + 1)
    assert bound <= width * _constant("kGrpStack")
    rng = np.random.default_rng(7)
    for p in (1.0, 0.95, 0.8, 0.6):
        assert _peak(levels, width, lambda d: rng.random() < p) <= bound
    for _ in range(8):
        at = rng.choice([0.5, 0.7, 0.9, 1.0], levels + 1)
        assert _peak(levels, width, lambda d: rng.random() < at[d]) <= bound
