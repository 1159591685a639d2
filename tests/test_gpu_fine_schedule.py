"""Large complex64 boxes: one right-hand side runs in finer tasks than several."""
import numpy as np
import pytest
import torch

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -23


@pytest.fixture(scope="module")
def case():
    nx, ny, nz = 128, 126, 30   # panels of 14, 14 and 10 planes and a remainder: boxes above and below 0.8 GB
    h = 1.0 / (nx + 1)
    c = wl.velocity_lens(nx, ny, nz, h)
    return Case(c, h, wl.omega_for_ppw(float(c.min()), 10.0, h), 10, 4, pad=10)


def handle(case, **kw):
    from paper_1204_0111_gb300 import psp
    return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                      pad=case.pad, leaf=case.leaf, pml_C=case.C, alpha=case.alpha, precision="c64", **kw)


@pytest.mark.parametrize("si", ["extended", "paper"])
def test_one_column_agrees_with_several_and_with_an_explicit_schedule(case, si):
    # sums of n <= 7000 products in another order differ by about sqrt(n) eps = 84 eps, in each of 2 m - 1 solves
    P, Q = handle(case, selective_inversion=si), handle(case, selective_inversion=si, sweep_level_tasks=304)
    r = torch.from_numpy(wl.random_vector(case.N, 2, seed=3)).cuda()
    both = P.apply(r, torch.empty_like(r))
    m = 2 * P.info()["panels"] - 1
    for q in (0, 1):
        one = r[q:q + 1].clone()
        a, b = P.apply(one, torch.empty_like(one))[0], Q.apply(one, torch.empty_like(one))[0]
        for x in (a, b):
            assert torch.linalg.vector_norm(x - both[q]) < 100 * m * EPS * torch.linalg.vector_norm(both[q])
        # with the explicit schedule one column and several run in the same tasks
        assert torch.linalg.vector_norm(Q.apply(r, torch.empty_like(r)) - both) == 0


def test_halves_and_the_tuner_keep_the_result(case):
    P = handle(case)
    r = torch.from_numpy(wl.random_vector(case.N, 1, seed=4)).cuda()
    ref = P.apply(r, torch.empty_like(r))
    u = r.clone()
    P.sweep_part(u, 0)
    P.sweep_part(u, 1)
    assert torch.equal(u, ref)
    t = P.tune_sweep(nrhs=1, reps=1)
    Q = handle(case, sweep_level_tasks=t["sweep_level_tasks"], sweep_min_rows=t["sweep_min_rows"],
               sweep_max_rows=t["sweep_max_rows"], sweep_claim_ahead=t["sweep_claim_ahead"])
    m = 2 * P.info()["panels"] - 1
    for H in (P, Q):
        out = H.apply(r, torch.empty_like(r))
        assert torch.linalg.vector_norm(out - ref) < 100 * m * EPS * torch.linalg.vector_norm(ref)
