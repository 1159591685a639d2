"""A tensor-core product that can never finish (test option: one operand block is announced and not copied): its bounded
waits give up, the setup reports PSP_ERR_TIMEOUT, and the device stays usable."""
import time

import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

from _cases import Case, random_velocity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c128", "c64"])
def test_a_stalled_product_is_reported_and_the_device_stays_usable(precision):
    import torch
    from oracle import sweep as osw
    from paper_1204_0111_gb300 import psp
    nx, ny, D = 33, 30, 4   # separators of 132, 120 and 64 rows: tensor-core products in both precisions
    h = 1.0 / (nx + 1)
    c = random_velocity(nx, ny, 2 * D, 5)
    case = Case(c, h, wl.omega_for_ppw(float(c.min()), 10.0, h), 1, D, pad=1)

    def handle(**kw):
        return psp.SweepingPreconditioner(torch.from_numpy(case.c).cuda(), case.h, case.omega, case.gamma, case.depth,
                                          pad=case.pad, leaf=case.leaf, precision=precision, **kw)

    t0 = time.monotonic()
    with pytest.raises(psp.PSPError) as e:
        handle(test_sweep_stall=2)
    assert e.value.name == "PSP_ERR_TIMEOUT"
    assert time.monotonic() - t0 < 60   # each wait gives up after about two seconds
    P = handle()
    r = wl.random_vector(case.N, 2, seed=1)
    out = P.apply(torch.from_numpy(r).cuda(), torch.empty((2, case.N), dtype=torch.complex128, device="cuda"))
    ref = osw.SweepingPreconditioner(case.oracle_problem(), case.depth, case.pad, case.leaf).apply(r)
    assert np.linalg.norm(out.cpu().numpy() - ref) < (1e-10 if precision == "c128" else 1e-4) * np.linalg.norm(ref)
