"""The form without inversion (one CTA substitutes through a whole front) with a front wider than shared memory."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [23, 24])   # one front of 12,167 rows (its vector fits) and of 13,824 (it does not)
def test_one_front_wider_than_shared_memory(n):
    # one panel without a pad: the preconditioner is J's inverse, so J applied to its result gives the input back
    import torch
    from paper_1204_0111_gb300 import psp
    h = 1.0 / (n + 1)
    c = wl.velocity_lens(n, n, n, h)
    P = psp.SweepingPreconditioner(torch.from_numpy(c).cuda(), h, wl.omega_for_ppw(float(c.min()), 10.0, h), 3, n, pad=0,
                                   leaf=n ** 3, selective_inversion="none")
    assert P.info()["panels"] == 1 and P.info()["fronts"] == 1
    r = torch.from_numpy(wl.random_vector(n ** 3, 3, seed=n)).cuda()
    x = P.apply(r, torch.empty_like(r))
    back = P.matvec(x, torch.empty_like(r), which=1)
    assert torch.linalg.vector_norm(back - r) < 1e-9 * torch.linalg.vector_norm(r)
