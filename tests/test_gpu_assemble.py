"""Front assembly in memory that held another model's fronts before: every entry is zeroed or written, whatever the alignment
of a CTA's 32 columns (odd and even front sizes, 8- and 16-byte elements) and the number of a child's rows (fewer and more
than the 32 probes of one search step)."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case, random_velocity

pytestmark = pytest.mark.gpu


def one_panel(nx, ny, D, leaf, seed):
    h = 1.0 / (max(nx, ny) + 1)
    c = random_velocity(nx, ny, D, seed)
    return Case(c, h, wl.omega_for_ppw(float(c.min()), 10.0, h), 1, D, pad=1, leaf=leaf)


# bounds: those of the other front comparisons, 1e-10 in complex128 and 1e-3 in complex64
@pytest.mark.parametrize("precision,bound", [("c128", 1e-10), ("c64", 1e-3)])
@pytest.mark.parametrize("si", ["extended", "two"])
@pytest.mark.parametrize("nx,ny,D,leaf", [(7, 5, 3, 16), (16, 16, 2, 16), (11, 9, 3, 16), (17, 15, 5, 16), (34, 31, 3, 64)])
def test_fronts_in_used_memory(nx, ny, D, leaf, si, precision, bound):
    import torch
    from oracle import sweep as osw
    from paper_1204_0111_gb300 import psp

    def handle(case):
        return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                          pad=case.pad, leaf=case.leaf, pml_C=case.C, alpha=case.alpha, faces=case.faces,
                                          precision=precision, selective_inversion=si)

    before = handle(one_panel(nx, ny, D, leaf, 3))
    before.close()
    case = one_panel(nx, ny, D, leaf, 7)
    O = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf)
    P = handle(case)
    for p in range(O.m):
        for f, fr in enumerate(O.fronts[p]):
            G, s, u = P.export_front(p, f)
            inv = np.linalg.inv(fr.L_TL)
            bot = fr.L_BL @ inv if si == "extended" else fr.L_BL
            low = np.tril(G[:s], -1) if s else G[:0]
            assert np.linalg.norm(low - np.tril(inv, -1)) <= bound * np.linalg.norm(inv)
            assert np.linalg.norm(np.diag(G[:s]) - fr.d) <= bound * np.linalg.norm(fr.d)
            if len(fr.L_BL):
                assert np.linalg.norm(G[s:] - bot) <= bound * np.linalg.norm(bot)
    P.close()
