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
    """device memory from PyTorch's caching allocator, NULL past cap live bytes
    and at call number fail_at"""

    def __init__(self, cap=None, fail_at=None):
        self.cap, self.live, self.peak, self.sizes, self.refused = cap, 0, 0, {}, 0
        self.fail_at, self.calls = fail_at, 0

    def alloc(self, nbytes, stream):
        self.calls += 1
        if self.calls == self.fail_at:
            self.refused += 1
            return None
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


def test_allocation_failure_at_every_allocation():
    """of a first request's admission and solve: it is refused for want of memory
    or solved with the same bits, nothing leaks, and a service that goes on
    (a failed admission does not stop it) solves the next request"""
    Uh = orc.gauge_start(DIMS, seed=30, eps=0.25)

    def ask(svc, gid, mem):
        t = svc.submit(gid, 0.152, (1, 2, 3, 0), 3)
        r = svc.wait(t)
        calls, mem.fail_at = mem.calls, None  # (the download has a buffer of its own)
        xs = []
        if r["status"] == lqcd.OK:
            xs = [lqcd.Field.borrowed(h, DIMS, lqcd.SPINOR_EVEN).download() for h in
                  (svc.solution(t, k)[0] for k in range(3))]
        svc.release(t)
        return r["status"], xs, calls

    U = lqcd.gauge_field(DIMS).upload(Uh)
    want, total, refused, solved, stopped, k = None, None, 0, 0, 0, 0
    while total is None or k <= total:
        mem = CappedAllocator(fail_at=k or None)
        lqcd.set_allocator(mem.alloc, mem.free)
        try:
            svc = lqcd.Service(lqcd.service_params(tol=TOL))
            gid = svc.add_gauge(U)
            status, xs, calls = ask(svc, gid, mem)
            if want is None:
                want, total = xs, calls
            assert status in (lqcd.OK, lqcd.ENOMEM) and (k == 0 or mem.refused == 1)
            if status == lqcd.OK:
                solved += 1
                assert all(np.array_equal(a, b) for a, b in zip(xs, want))
            else:
                refused += 1
                try:
                    status, xs, _ = ask(svc, gid, mem)
                    assert status == lqcd.OK and all(np.array_equal(a, b) for a, b in zip(xs, want))
                except lqcd.LqcdError as e:
                    assert e.status == lqcd.ENOMEM  # the solver's tables: the service has stopped
                    stopped += 1
            svc.close()
            assert mem.live == 0, k
        finally:
            lqcd.set_allocator(None, None)
        k += 1
    assert refused > 10 and solved > 10 and stopped < 6
