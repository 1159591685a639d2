"""The complex128 front products on the tensor cores where a product's columns differ by many orders (PML amplitudes of
1e4 .. 1e6 times the usual one, frequencies near zero: pivots of very different sizes).

A product C = A B^T in 64-bit arithmetic has entries wrong by at most about n 2^-53 P_ij, P = |A| |B|^T, n terms.  The digit
products promise that relative to sqrt(max_j P_ij max_i P_ij), which is no smaller; the bound below, 8 n 2^-53 of it, covers
the three real products a complex one is made of, their sums, and both sides of a comparison.  Only fronts without
children are compared, whose inputs are the same on both sides."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case, random_velocity

pytestmark = pytest.mark.gpu


def case_of(C, omega, leaf):
    nx, ny, D = 18, 16, 6
    h = 1.0 / (nx + 1)
    c = random_velocity(nx, ny, D, 7)
    return Case(c, h, omega or wl.omega_for_ppw(float(c.min()), 10.0, h), 1, D, pad=1, leaf=leaf, C=C)


def handle(case, **kw):
    import torch
    from paper_1204_0111_gb300 import psp
    return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                      pad=case.pad, leaf=case.leaf, pml_C=case.C, alpha=case.alpha, faces=case.faces, **kw)


def leaves(case, P):
    """(front, oracle's factor of it) of the fronts without children that the tensor cores take."""
    from oracle import sweep as osw
    from paper_1204_0111_gb300 import psp
    O = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf)
    sns = psp.parse_symbolic(P.symbolic(0))[1]
    parents = {sn[2] for sn in sns}
    out = [(f, fr) for f, fr in enumerate(O.fronts[0]) if f not in parents and len(fr.d) >= 16 and fr.L_BL.shape[0] >= 16]
    assert out
    return out


def worst(diff, A, B, rows=slice(None)):
    """Largest entry of diff (the product's given rows) relative to sqrt(row maximum x column maximum) of |A| |B|^T, in
    units of the bound."""
    P = np.abs(A) @ np.abs(B).T
    scale = np.sqrt(P.max(1)[rows, None] * P.max(0)[None, :])
    return np.max(np.abs(diff) / np.where(scale > 0, scale, 1.0)) / (8 * A.shape[1] * 2.0 ** -53)


CASES = [(4.0, None), (4e4, None), (4e6, None), (4e3, 1e-4)]


@pytest.mark.parametrize("C,omega", CASES)
@pytest.mark.parametrize("leaf", [100, 250])
def test_z_of_columns_of_very_different_size(C, omega, leaf):
    case = case_of(C, omega, leaf)
    P, Q = handle(case, selective_inversion="paper"), handle(case, selective_inversion="paper", tensor_cores=False)
    for f, fr in leaves(case, P):
        s = len(fr.d)
        G, H = P.export_front(0, f)[0], Q.export_front(0, f)[0]
        assert np.array_equal(G[:s], H[:s])   # up to here both sides computed the same
        inv = np.tril(G[:s], -1) + np.eye(s)
        d = np.diag(G[:s])
        FBL = (fr.L_BL * fr.d) @ fr.L_TL.T
        assert worst((G[s:] - H[s:]) * d, FBL, inv) < 1, f


@pytest.mark.parametrize("C,omega", CASES)
@pytest.mark.parametrize("leaf", [100, 250, 700])
def test_m_bl_of_columns_of_very_different_size(C, omega, leaf):
    # M_BL = L_BL inv(L_TL) against the product of the factors that the paper's form keeps, in long double
    case = case_of(C, omega, leaf)
    P, Q = handle(case), handle(case, selective_inversion="paper")
    for f, fr in leaves(case, P):
        s = len(fr.d)
        G, H = P.export_front(0, f)[0], Q.export_front(0, f)[0]
        assert np.array_equal(G[:s], H[:s])
        inv = np.tril(G[:s], -1) + np.eye(s)
        rows = np.linspace(0, len(G) - s - 1, 24).astype(int)
        ref = H[s:][rows].astype(np.clongdouble) @ inv.astype(np.clongdouble)
        assert worst((G[s:][rows] - ref).astype(np.complex128), H[s:], inv.T, rows) < 1, f
