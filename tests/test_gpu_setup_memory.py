"""The memory a complex128 setup takes for its temporaries: the caller's cap holds, with the same factors, and a pool that is
enough for a setup on CUDA cores is enough for the default one."""
import numpy as np
import pytest

from paper_1204_0111_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def handle(w, **kw):
    import torch
    from paper_1204_0111_gb300 import psp
    return psp.SweepingPreconditioner(torch.from_numpy(w.c).cuda(), w.h, w.omega, w.gamma, w.panel_depth, pad=w.pad, leaf=w.leaf,
                                      pml_C=w.pml_C, alpha=w.alpha, **kw)


class Pool:
    """torch's caching allocator, refusing what would pass a limit."""

    def __init__(self, limit):
        self.limit, self.live, self.sum, self.peak, self.refused = limit, {}, 0, 0, 0

    def alloc(self, n):
        import torch
        if self.sum + n > self.limit:
            self.refused += 1
            return 0
        p = torch.cuda.caching_allocator_alloc(n)
        self.live[p] = n
        self.sum += n
        self.peak = max(self.peak, self.sum)
        return p

    def free(self, p):
        import torch
        torch.cuda.caching_allocator_delete(p)
        self.sum -= self.live.pop(p)


def fronts_of(P):
    return [P.export_front(i, f)[0] for i in range(0, P.info()["panels"], 3) for f in (0, 7, 40, 90, 200, 550, 571, 572)]


# the widest fronts of a 48^3 lens: 576 rows (the root), 276 with a struct of 576; on CUDA cores they need 6.3 MiB (10.2 with
# two inverses), their digits in one piece up to 18: pieces of fewer columns and of fewer rows, and everything at once
@pytest.mark.parametrize("mb,si", [(m, f) for f in ("extended", "paper", "two") for m in (7, 8, 11, 16, 64) if f != "two" or m > 10])
def test_cap_on_temporaries_holds_and_does_not_change_the_factors(mb, si):
    w = wl.cube_lens(48)
    P, Q = handle(w, selective_inversion=si), handle(w, selective_inversion=si, setup_temp_mb=mb)
    for a, b in zip(fronts_of(P), fronts_of(Q)):
        assert np.array_equal(a, b)
    assert 0 < Q.stats()["host:alloc_work"]["bytes"] <= mb << 20
    assert Q.stats()["k_oz_gemm"]["launches"] > 0
    if si == "two":
        assert np.array_equal(P.export_second_inverse(3, 572), Q.export_second_inverse(3, 572))


@pytest.mark.parametrize("si", ["extended", "paper"])
@pytest.mark.parametrize("mb", [0, 8])
def test_a_pool_that_holds_a_setup_on_cuda_cores_holds_the_default_one(mb, si):
    w = wl.cube_lens(48)
    kw = dict(setup_temp_mb=mb, selective_inversion=si)
    wide = Pool(1 << 40)
    P = handle(w, tensor_cores=False, allocator=(wide.alloc, wide.free), **kw)
    P.close()
    tight = Pool(wide.peak)
    Q = handle(w, allocator=(tight.alloc, tight.free), **kw)
    ref = handle(w, selective_inversion=si)
    assert tight.peak <= wide.peak
    for a, b in zip(fronts_of(Q), fronts_of(ref)):
        assert np.linalg.norm(a - b) < 1e-12 * np.linalg.norm(b)
    Q.close()
    assert not tight.live


def test_without_any_room_the_setup_reports_it():
    from paper_1204_0111_gb300 import psp
    w = wl.cube_lens(32)
    pool = Pool(1 << 40)
    P = handle(w, allocator=(pool.alloc, pool.free))
    fb = P.info()["factor_bytes"]
    P.close()
    small = Pool(fb + (1 << 20))   # room for the factors, none for the temporaries
    with pytest.raises(psp.PSPError) as e:
        handle(w, allocator=(small.alloc, small.free))
    assert e.value.name == "PSP_ERR_OOM" and not small.live
