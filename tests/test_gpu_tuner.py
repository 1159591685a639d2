"""The sweep's autotuner times a schedule once: CTAs per SM beyond what fits, and groups of more columns than a pass carries,
come to a launch that it has already timed."""
import pytest
import torch

from paper_1204_0111_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,groups", [("c128", 2), ("c64", 3)])   # 1, 2 (and 4) columns besides the default 4 (8)
def test_equal_launches_are_timed_once(precision, groups):
    from paper_1204_0111_gb300 import psp
    w = wl.cube_lens(24)
    P = psp.SweepingPreconditioner(torch.from_numpy(w.c).cuda(), w.h, w.omega, w.gamma, w.panel_depth, pad=w.pad, leaf=w.leaf,
                                   pml_C=w.pml_C, alpha=w.alpha, precision=precision)
    t = P.tune_sweep(nrhs=8, reps=1)
    # the schedule at hand, two other caps on rows, four other level counts, the groups, four other floors, one other claim
    assert t["candidates"] == 1 + 2 + 4 + groups + 4 + 1
