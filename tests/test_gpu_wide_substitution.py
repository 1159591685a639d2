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


# fronts of one 32-column block and of several, at the edges of the block and of the 8 and 16 columns read ahead in it
@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("rows", [(1, 1, 1), (7, 1, 1), (8, 1, 1), (3, 3, 1), (15, 1, 1), (4, 2, 2), (17, 1, 1), (31, 1, 1), (4, 4, 2),
                                  (11, 3, 1), (7, 7, 1), (8, 4, 2), (13, 5, 1), (6, 5, 4), (8, 4, 4), (43, 3, 1)])
@pytest.mark.parametrize("nrhs", [1, 3, 8])
def test_one_front_at_the_edges_of_its_blocks(nrhs, rows, precision):
    import torch
    from paper_1204_0111_gb300 import psp
    nx, ny, nz = rows
    h = 1.0 / (max(rows) + 1)
    c = wl.velocity_lens(nx, ny, nz, h)
    P = psp.SweepingPreconditioner(torch.from_numpy(c).cuda(), h, wl.omega_for_ppw(float(c.min()), 10.0, h), 1, nz, pad=0,
                                   leaf=nx * ny * nz, selective_inversion="none", precision=precision)
    assert P.info()["fronts"] == 1
    r = torch.from_numpy(wl.random_vector(nx * ny * nz, nrhs, seed=nx)).cuda()
    x = P.apply(r, torch.empty_like(r))
    back = P.matvec(x, torch.empty_like(r), which=1)
    assert torch.linalg.vector_norm(back - r) < (1e-11 if precision == "c128" else 1e-3) * torch.linalg.vector_norm(r)
