"""The launch shapes that the autotuner tries hold those that the kernels take when none is set, as include/at.h states them
at at_set_launch: a solver that was tuned can run in the shape it had before."""
import os
import re

from paper_1702_00496_gb300 import autotune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_default_shapes_are_candidates():
    text = open(os.path.join(ROOT, "include", "at.h")).read().split("int at_set_launch(")[0].split("/* Launch shape")[-1]
    found = re.search(r"Defaults (\d+) and (\d+); (\d+) and (\d+) for 1D", text)
    assert found, text
    a, b, c, d = (int(v) for v in found.groups())
    assert {(a, b), (c, d)} <= set(autotune.FORWARD_CANDIDATES)
    assert len(set(autotune.FORWARD_CANDIDATES)) == len(autotune.FORWARD_CANDIDATES)
    assert all(t in (128, 256, 512) and 1 <= n <= 64 for t, n in autotune.FORWARD_CANDIDATES)
