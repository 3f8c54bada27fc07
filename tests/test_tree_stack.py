"""CPU: the traversal stack of tree gravity holds every walk.  The rule of the
walk (four cells off the top, their opened children in lane order in their
place) is run over trees of every depth with many ways to open cells, and the
places it uses are compared with the kernel's bound."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_11322_gb300", "csrc")


def constant(name, path):
    with open(os.path.join(CSRC, path)) as f:
        return int(re.search(r"constexpr int " + name + r" = (\d+);", f.read()).group(1))


PARTS = constant("kTreeParts", "dem_internal.h")
MAX_DEPTH = constant("kTreeMaxDepth", "dem_internal.h")
SPLIT = constant("kSplitL", "kernels_tree.cu")


def places(depth):
    return 64 // PARTS + 31 * (depth - 1 - SPLIT)


def test_the_kernel_sizes_its_stack_by_the_bound():
    with open(os.path.join(CSRC, "kernels_tree.cu")) as f:
        assert "kTreeStack = 64 / kTreeParts + 31 * (kTreeMaxDepth - 1 - kSplitL);" in f.read()


def walk(depth, opened):
    """Highest stack of one walk; opened(level): how many of a cell's 8 children are opened again."""
    # the first round tests the walk's own cells, which are leaves in a tree of depth SPLIT
    stack = [SPLIT] * (64 // PARTS) if SPLIT < depth else []
    high = len(stack)
    while stack:
        taken = [stack.pop() for _ in range(min(4, len(stack)))]     # the top one first: lanes 0..7
        for level in taken:
            if level + 1 < depth:
                stack += [level + 1] * opened(level + 1)
        high = max(high, len(stack))
    return high


@pytest.mark.parametrize("depth", range(SPLIT, MAX_DEPTH + 1))
def test_walks_stay_inside_the_stack(depth):
    rng = random.Random(depth)
    bound = places(depth) if depth > SPLIT else 0
    assert walk(depth, lambda level: 8) <= bound
    for trial in range(60):
        share = rng.random()
        few = rng.randint(0, 3)
        ways = (lambda level: 8 if rng.random() < share else few,
                lambda level: rng.randint(0, 8),
                lambda level: 8 if level < depth - 1 or rng.random() < share else few,
                lambda level: 8 - few if level % 2 else 8)
        for opened in ways:
            assert walk(depth, opened) <= bound
