"""The autotuner's candidates and choice (no GPU: the timing is the library's)."""
import os
import re

import pytest

from paper_2311_10048_gb300 import tune

CSRC = os.path.join(os.path.dirname(tune.__file__), "csrc")


@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "tf32", "bf16x6", "bf16x10", "bf16x15"])
def test_the_untuned_schedule_is_always_a_candidate(prec):
    cap = int(re.search(r"kGroupCap = (\d+);",
                        open(os.path.join(CSRC, "lno_ot.cu")).read()).group(1))
    assert tune.DEFAULT == (0, cap)
    rows = tune.candidates(prec)
    assert tune.DEFAULT in rows and len(set(rows)) == len(rows)
    slices = {"fp64": 1, "bf16x3": 2, "tf32": 2, "bf16x6": 3, "bf16x10": 3, "bf16x15": 5}[prec]
    assert all(bn % 16 == 0 and 0 <= bn <= min(256, 512 // slices) and 1 <= g <= cap
               for bn, g in rows)


def test_a_row_replaces_the_default_only_by_a_margin():
    t = {(0, 1024): 10.0, (0, 64): 12.0, (96, 1024): 9.95}
    assert tune.pick(t) == (0, 1024)
    t[(96, 1024)] = 9.0
    assert tune.pick(t) == (96, 1024)
