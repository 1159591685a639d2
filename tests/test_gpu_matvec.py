"""The 7-point products over every combination of axes with and without PML, in boxes whose rows are shorter than, equal to
and longer than a warp, so that warps meet each combination and mixtures of them."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case, random_velocity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("faces", [0, 1, 2, 4, 8, 16, 32, 3, 12, 48, 21, 63])
@pytest.mark.parametrize("dims", [(1, 1, 5), (7, 5, 9), (32, 3, 12), (33, 31, 11), (70, 9, 10)])
def test_products_match_the_oracle_and_columns_keep_their_bits(dims, faces):
    import torch
    from oracle import discretize as dz
    from paper_1204_0111_gb300 import psp
    nx, ny, nz = dims
    h = 1.0 / (max(dims) + 1)
    case = Case(random_velocity(nx, ny, nz, 3), h, 2 * np.pi / (10 * h), 3 if faces else 0, 4, pad=2, faces=faces)
    p = case.oracle_problem()
    P = psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth, pad=case.pad,
                                   leaf=case.leaf, pml_C=case.C, alpha=case.alpha, faces=case.faces)
    x = wl.random_vector(case.N, 3, seed=4)
    xd = torch.from_numpy(x).cuda()
    for which, A in ((0, dz.operator_A(p)), (1, dz.operator_J(p))):
        y = P.matvec(xd, torch.empty_like(xd), which=which)
        ref = (A @ x.T).T
        # at most 8 products and sums of a few roundings each per entry
        assert np.linalg.norm(y.cpu().numpy() - ref) < 1e-14 * np.linalg.norm(ref)
        for q in range(3):
            one = xd[q:q + 1].clone()
            assert torch.equal(P.matvec(one, torch.empty_like(one), which=which)[0], y[q])
