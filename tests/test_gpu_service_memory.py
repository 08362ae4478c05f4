"""The solve service where device memory is short: the further sets of float-float
temporaries are made only where there is room, and given back when another
request's admission needs theirs; what fits with one set per gauge field is
solved, with the same bits."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)
VH = 2048
SET = 3 * 192 * VH  # bytes of one set: two even and one odd float-float spinor
TOL = 1e-10


class CappedAllocator:
    """device memory from PyTorch's caching allocator, NULL past cap live bytes"""

    def __init__(self, cap=None):
        self.cap, self.live, self.peak, self.sizes, self.refused = cap, 0, 0, {}, 0

    def alloc(self, nbytes, stream):
        if self.cap is not None and self.live + nbytes > self.cap:
            self.refused += 1
            return None
        p = torch.cuda.caching_allocator_alloc(nbytes)
        self.sizes[p] = nbytes
        self.live += nbytes
        self.peak = max(self.peak, self.live)
        return p

    def free(self, ptr, stream):
        self.live -= self.sizes.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)


def run(Uh, order, cap=None):
    """requests on the gauge fields of order, one after another, all kept"""
    mem = CappedAllocator(cap)
    lqcd.set_allocator(mem.alloc, mem.free)
    try:
        svc = lqcd.Service(lqcd.service_params(tol=TOL))
        fields = [lqcd.gauge_field(DIMS).upload(u) for u in Uh]
        ids = [svc.add_gauge(U) for U in fields]
        out = []
        for g in order:
            t = svc.submit(ids[g], 0.152, (1, 2, 3, g), 12)
            r = svc.wait(t)
            assert r["status"] == lqcd.OK, (r, mem.refused)
            assert r["true_rel_res_max"] <= TOL
            xs = []
            for k in range(12):
                e, o = svc.solution(t, k)
                xs.append(lqcd.Field.borrowed(e, DIMS, lqcd.SPINOR_EVEN).download())
                xs.append(lqcd.Field.borrowed(o, DIMS, lqcd.SPINOR_ODD).download())
            out.append((r["iters"], xs))
        svc.close()
        for U in fields:
            U.free()
        assert mem.live == 0
        return out, mem
    finally:
        lqcd.set_allocator(None, None)


def same(a, b):
    return all(x[0] == y[0] and all(np.array_equal(p, q) for p, q in zip(x[1], y[1])) for x, y in zip(a, b))


@pytest.mark.parametrize("order,dropped", [([0], 3.99), ([0], 4), ([0], 4.02), ([0], 11), ([0, 1], 15), ([0, 1], 22),
                                           ([0, 1, 0], 22)])
def test_requests_that_fit_with_fewer_sets(order, dropped):
    """dropped: sets (of the 12 per gauge field) that the cap leaves no room for;
    a fraction more or less, room for the solver's tables or none beside them"""
    Uh = [orc.gauge_start(DIMS, seed=30 + k, eps=0.25) for k in range(1 + max(order))]
    free, mem = run(Uh, order)
    assert mem.refused == 0
    got, capped = run(Uh, order, cap=mem.peak - int(dropped * SET))
    assert capped.refused > 0 and same(free, got)
