"""Task lists of the setup: with many groups of fronts each list is refilled while the groups before are still being
uploaded and factored.  The factors of every such setup are those of a setup with one group per tree level, bit for bit."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c128", "c64"])
def test_refilled_lists_give_the_same_factors(precision):
    import torch
    from paper_1204_0111_gb300 import psp
    w = wl.cube_lens(48)
    c = torch.from_numpy(w.c).cuda()

    def handle(**kw):
        return psp.SweepingPreconditioner(c, w.h, w.omega, w.gamma, w.panel_depth, pad=w.pad, leaf=w.leaf, pml_C=w.pml_C,
                                          alpha=w.alpha, precision=precision, **kw)

    P = handle()
    fronts = [(i, f) for i in range(P.info()["panels"]) for f in (0, 7, 40, 90)]
    ref = [P.export_front(i, f)[0] for i, f in fronts]
    for mb in (32, 16, 16):   # tens of groups each
        Q = handle(setup_temp_mb=mb)
        for (i, f), g in zip(fronts, ref):
            assert np.array_equal(Q.export_front(i, f)[0], g), (mb, i, f)
        Q.close()
