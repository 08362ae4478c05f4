"""Which solves take the solver's resident kernel, and what it does at its limits:
with the boundary sign and the anisotropic weights it has the bits of the
kernel-by-kernel path (taken while a hopping-term class is timed); a launch that
returns after a few iterations is resumed without a trace; a barrier whose wait
runs out ends the solve with LQCD_ETIMEOUT and the next solve is whole."""
import numpy as np
import pytest

from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu

# blocks of 128 even sites (FP64: 32).  (4,4,6,10) FP64: 15, ragged, a cluster of
# 16 with an empty block; (2,2,10,26) FP64: 17, ragged, the first size of the
# barrier over the grid; (14,14,14,14) FP64: 601, ragged, (16,16,16,36): 576, near
# the 608 that run at once; (14,14,14,16) FP64: 686 and (20,20,20,20): 625, above
RESIDENT = [("f64", (4, 4, 4, 4)), ("f64", (4, 4, 6, 10)), ("f64", (2, 2, 10, 26)), ("f64", (14, 14, 14, 14)),
            ("f32", (4, 4, 6, 10)), ("f16n", (2, 2, 10, 26)), ("bf16", (6, 6, 10, 12)), ("f32", (16, 16, 16, 36)),
            ("f16n", (16, 16, 16, 36)), ("bf16", (16, 16, 16, 36))]
BY_KERNEL = [("f64", (14, 14, 14, 16)), ("f32", (20, 20, 20, 20)), ("f16n", (20, 20, 20, 20)),
             ("bf16", (20, 20, 20, 20))]


@pytest.fixture(autouse=True)
def default_limits():
    yield
    lqcd.solver_limits()


class Problem:
    def __init__(self, dims, prec, **geo):
        self.dims, self.geo, self.sloppy = dims, geo, lqcd.PREC_NAMES[prec]
        self.U = lqcd.gauge_field(dims, **geo)
        lqcd.gauge_start(self.U, 5, 0.2)
        self.b = lqcd.spinor_field(dims, 0, **geo)
        lqcd.eta_refresh(self.b, 6, 0)
        self.Us = None if prec == "f64" else lqcd.gauge_field(dims, self.sloppy, **geo).copy_from(self.U)
        self.prm = lqcd.cg_params(tol=1e-10, sloppy=self.sloppy, delta=0.05)

    def solve(self, check=True):
        """the outcome with the solution's bits, and the number of launches"""
        x = lqcd.spinor_field(self.dims, 0, **self.geo)
        n0 = lqcd.launch_count()
        rc, info = lqcd.cg_solve(x, self.U, self.b, 0.15, self.prm, U_sloppy=self.Us, check=check)
        n = lqcd.launch_count() - n0
        return (rc, info.iters, info.restarts, info.true_rel_res, x.download().tobytes()), n

    def by_kernel(self):
        lqcd.kernel_timers(True)
        try:
            return self.solve()
        finally:
            lqcd.kernel_timers(False)


@pytest.mark.parametrize("prec,dims", RESIDENT + BY_KERNEL)
def test_the_path_taken(prec, dims):
    p = Problem(dims, prec)
    got, n = p.solve()
    ref, n_ref = p.by_kernel()
    assert got[0] == lqcd.OK and got == ref
    if (prec, dims) in RESIDENT:
        assert n < n_ref - 2 * got[1]  # five launches per iteration saved
    else:
        assert n == n_ref


@pytest.mark.parametrize("prec", ["f64", "f32", "f16n", "bf16"])
@pytest.mark.parametrize("geo", [dict(t_bc=1), dict(t_bc=-1, aniso=(2.5, 1.2)), dict(t_bc=1, aniso=(2.5, 1.2))])
@pytest.mark.parametrize("dims", [(4, 4, 6, 10), (6, 6, 10, 12)])
def test_boundary_and_anisotropy_bitwise(prec, geo, dims):
    p = Problem(dims, prec, **geo)
    got, n = p.solve()
    ref, n_ref = p.by_kernel()
    assert got[0] == lqcd.OK and got == ref and n < n_ref


@pytest.mark.parametrize("prec", ["f64", "f32", "f16n", "bf16"])
@pytest.mark.parametrize("dims", [(4, 4, 6, 10), (6, 6, 10, 20)])  # a cluster, and (29 blocks) the barrier over the grid
@pytest.mark.parametrize("iterations", [1, 3])
def test_launches_of_few_iterations(prec, dims, iterations):
    p = Problem(dims, prec)
    ref, n_ref = p.solve()
    lqcd.solver_limits(iterations=iterations)
    got, n = p.solve()
    assert got == ref and n > n_ref


@pytest.mark.parametrize("prec", ["f64", "f32", "f16n", "bf16"])
def test_barrier_that_gives_up(prec):
    p = Problem((16, 16, 16, 16), prec) if prec != "f64" else Problem((8, 8, 8, 16), prec)  # 256, 128 blocks
    ref, _ = p.solve()
    lqcd.solver_limits(polls=1)
    got, _ = p.solve(check=False)
    assert got[0] == lqcd.ETIMEOUT
    with pytest.raises(lqcd.LqcdError, match="barrier gave up"):
        p.solve()
    lqcd.solver_limits()
    assert p.solve()[0] == ref


@pytest.mark.parametrize("prec,dims", BY_KERNEL)
def test_refused_launch_goes_kernel_by_kernel(prec, dims):
    """a grid that the device does not hold at once (or a process with a part of
    its SMs does not): the runtime refuses the cooperative launch"""
    p = Problem(dims, prec)
    ref, n_ref = p.solve()
    lqcd.solver_limits(blocks=1 << 20)
    got, n = p.solve()
    assert got == ref and n == n_ref


def test_limits_are_checked():
    for bad in ((-1, 0, 0), (0, -1, 0), (0, 0, -1)):
        with pytest.raises(lqcd.LqcdError):
            lqcd.solver_limits(*bad)
