"""The persistent sweep at the edges of its task shapes: right-hand-side groups of every width (full, partial,
vectors too short for 16-byte loads), fronts wider than one staged chunk, than the index words a task slot holds and
than a task, and boxes whose consecutive panels have different trees."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case

pytestmark = pytest.mark.gpu

EPS = {"c128": 2.0 ** -52, "c64": 2.0 ** -23}


def handle(case, **kw):
    import torch
    from paper_1204_0111_gb300 import psp
    return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                      pad=case.pad, leaf=case.leaf, pml_C=case.C, alpha=case.alpha, faces=case.faces, **kw)


def box(nx, ny, nz, gamma=3, depth=4, pad=3):
    h = 1.0 / (max(nx, ny, nz) + 1)
    c = wl.velocity_lens(nx, ny, nz, h)
    return Case(c, h, wl.omega_for_ppw(float(c.min()), 10.0, h), gamma, depth, pad=pad)


@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("si", ["extended", "paper", "two", "none"])
@pytest.mark.parametrize("nrhs", [2, 3, 5, 8, 9])
def test_every_group_width_gives_each_column_its_own_bits(nrhs, si, precision):
    # a column's sums run in the same order whatever columns share its pass
    import torch
    case = box(17, 15, 19)
    P = handle(case, precision=precision, selective_inversion=si)
    r = torch.from_numpy(wl.random_vector(case.c.size, nrhs, seed=nrhs)).cuda()
    out = P.apply(r, torch.empty_like(r))
    for q in range(nrhs):
        one = r[q:q + 1].clone()
        assert torch.equal(P.apply(one, torch.empty_like(one))[0], out[q]), q


@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("dims,depth,pad", [((70, 66, 24), 5, 8), ((90, 88, 40), 12, 16)])
def test_wide_fronts_in_chunks(dims, depth, pad, precision):
    # separators of about 1000 and 2500 rows: a group of eight stages its vector in chunks, one column does not.  Sums
    # of n products in another order differ by about sqrt(n) eps (n <= 7500 rows: 87 eps), in each of 2 m - 1 solves
    import torch
    case = box(*dims, gamma=4, depth=depth, pad=pad)
    P = handle(case, precision=precision)
    r = torch.from_numpy(wl.random_vector(case.c.size, 8, seed=1)).cuda()
    out = P.apply(r, torch.empty_like(r))
    for q in (0, 7):
        one = r[q:q + 1].clone()
        ref = P.apply(one, torch.empty_like(one))[0]
        m = 2 * P.info()["panels"] - 1
        assert torch.linalg.vector_norm(out[q] - ref) < 100 * m * EPS[precision] * torch.linalg.vector_norm(ref)


@pytest.mark.parametrize("nz", [8, 9, 13, 15])
def test_consecutive_panels_of_different_depths(nz):
    # the last panel's remainder gives its box another tree than the panel below it
    import torch
    from oracle import sweep as osw
    case = box(15, 14, nz, gamma=2, depth=3, pad=4)
    O = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf)
    r = wl.random_vector(case.c.size, 3, seed=nz)
    P = handle(case)
    out = P.apply(torch.from_numpy(r).cuda(), torch.empty((3, case.c.size), dtype=torch.complex128, device="cuda"))
    ref = O.apply(r)
    assert np.linalg.norm(out.cpu().numpy() - ref) < 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("si", ["extended", "paper", "two"])
@pytest.mark.parametrize("min_rows", [2, 4, 8, 64])
def test_narrowest_tasks(min_rows, si, precision):
    # tasks of 2 rows or columns: several lanes share a row, all warps share a block of columns
    import torch
    from oracle import sweep as osw
    case = box(19, 14, 13)
    O = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf)
    r = wl.random_vector(case.c.size, 3, seed=min_rows)
    P = handle(case, precision=precision, selective_inversion=si, sweep_min_rows=min_rows, sweep_level_tasks=2432)
    out = P.apply(torch.from_numpy(r).cuda(), torch.empty((3, case.c.size), dtype=torch.complex128, device="cuda"))
    ref = O.apply(r)
    assert np.linalg.norm(out.cpu().numpy() - ref) < (1e-10 if precision == "c128" else 1e-4) * np.linalg.norm(ref)
