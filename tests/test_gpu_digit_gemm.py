"""The complex128 front products on the tensor cores (exact digit products) against the FP64 units' and against the
oracle's factors, at the edges of their 128 x 32 tiles, blocks of 16 k and accumulations of 128 k, and with front
entries of very different sizes."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case, random_velocity

pytestmark = pytest.mark.gpu


def handle(case, **kw):
    import torch
    from paper_1204_0111_gb300 import psp
    return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                      pad=case.pad, leaf=case.leaf, pml_C=case.C, alpha=case.alpha, faces=case.faces, **kw)


def box(nx, ny, D, high=1.0, leaf=64):
    # one panel (every plane in it): fronts of (width x D) separators
    h = 1.0 / (max(nx, ny) + 1)
    c = random_velocity(nx, ny, D, 7)
    c[:, ny // 3, :] *= high   # a fast slab: rows of F of another size
    return Case(c, h, wl.omega_for_ppw(float(c.min()), 10.0, h), 1, D, pad=1, leaf=leaf)


# separators of nx D and ny D rows and structs of up to 2 (nx + ny) D: s and u just below, at and above 16, 32, 128 and 144
@pytest.mark.parametrize("nx,ny,D,leaf", [(7, 5, 3, 16), (16, 16, 2, 16), (17, 15, 8, 64), (18, 16, 8, 64), (33, 32, 4, 64),
                                          (43, 41, 3, 64), (36, 36, 4, 64), (19, 17, 16, 64), (30, 26, 16, 64)])
@pytest.mark.parametrize("si", ["extended", "paper", "two"])
def test_fronts_match_the_oracle_as_closely_as_fp64_products(nx, ny, D, leaf, si):
    from oracle import sweep as osw
    case = box(nx, ny, D, leaf=leaf)
    O = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf)
    P, Q = handle(case, selective_inversion=si, collect_stats=1), handle(case, selective_inversion=si, tensor_cores=False)
    wide = any(len(fr.d) >= 16 and fr.L_BL.shape[0] >= 16 for p in range(O.m) for fr in O.fronts[p])
    assert wide == any(k == "k_oz_gemm" and v["launches"] > 0 for k, v in P.stats().items())
    worst = {"digits": 0.0, "fp64": 0.0}
    for p in range(O.m):
        for f, fr in enumerate(O.fronts[p]):
            u = fr.L_BL.shape[0]
            if u == 0:
                continue
            bot = fr.L_BL if si != "extended" else np.linalg.solve(fr.L_TL.T, fr.L_BL.T).T
            for name, hdl in (("digits", P), ("fp64", Q)):
                G, s, _ = hdl.export_front(p, f)
                worst[name] = max(worst[name], np.linalg.norm(G[s:] - bot) / np.linalg.norm(bot))
    # both carry the same rounding of the assembled fronts; the digit products themselves err less (0.2 - 0.6 of FP64)
    assert worst["digits"] < 2 * worst["fp64"] + 1e-15, worst
    assert worst["digits"] < 1e-10


@pytest.mark.parametrize("high", [1e-3, 1e3, 1e10])
def test_rows_of_very_different_size(high):
    # c^2 in the diagonal of F: entries 1e-20 .. 1e6 apart share a front, each row with its own scale
    import torch
    case = box(24, 22, 6, high=high)
    case.omega = 30.0
    P, Q = handle(case), handle(case, tensor_cores=False)
    r = torch.from_numpy(wl.random_vector(case.N, 2, seed=2)).cuda()
    a, b = P.apply(r, torch.empty_like(r)), Q.apply(r, torch.empty_like(r))
    assert torch.linalg.vector_norm(a - b) < 1e-10 * torch.linalg.vector_norm(b)
    G, H = P.export_front(0, 3)[0], Q.export_front(0, 3)[0]
    assert np.linalg.norm(G - H) < 1e-10 * np.linalg.norm(H)


def test_wave_speed_that_is_not_a_number_is_reported_or_carried():
    # a NaN in a front's rows stays a NaN in what it touches, as with FP64 products
    import torch
    case = box(24, 22, 6)
    case.c[2, 5, 5] = np.nan
    out = []
    for tc in (True, False):
        P = handle(case, tensor_cores=tc)
        r = torch.from_numpy(wl.random_vector(case.N, 1, seed=2)).cuda()
        out.append(torch.isnan(torch.view_as_real(P.apply(r, torch.empty_like(r)))).any().item())
    assert out[0] == out[1]
