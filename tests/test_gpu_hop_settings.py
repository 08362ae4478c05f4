"""A solve keeps the hopping-term form and block size that it started with: another
thread that switches the form or loads a tuned table meanwhile does not reach it,
so its solution is bitwise that of one of the settings (the form and the block
size set the order of its sums)."""
import threading

import numpy as np
import pytest

from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu

DIMS = (20, 20, 20, 20)  # 625 blocks of 128 sites: iterated kernel by kernel


def test_solve_ignores_settings_changed_while_it_runs(tmp_path):
    U = lqcd.gauge_field(DIMS)
    lqcd.gauge_start(U, 5, 0.2)
    b = lqcd.spinor_field(DIMS, 0)
    lqcd.eta_refresh(b, 6, 0)
    Us = lqcd.gauge_field(DIMS, lqcd.F16N).copy_from(U)
    prm = lqcd.cg_params(tol=1e-10, maxiter=1000, sloppy=lqcd.F16N, delta=0.05)
    tables = {}
    for block in (64, 128, 256):
        tables[block] = tmp_path / f"{block}.txt"
        tables[block].write_text("dslash_f16n {} {} {} {} {} 1.0 1\n".format(*DIMS, block))

    def solve():
        x = lqcd.spinor_field(DIMS, 0)
        rc, info = lqcd.cg_solve(x, U, b, 0.15, prm, U_sloppy=Us)
        return rc, info.iters, x.download().tobytes()

    stop = threading.Event()

    def switch():
        k = 0
        while not stop.is_set():
            lqcd.autotune_load(tables[(64, 256, 128)[k % 3]])
            lqcd.dslash_form(lqcd.DSLASH_PACKED if k % 2 else lqcd.DSLASH_PREFETCH)
            k += 1

    form = lqcd.dslash_form()
    t = threading.Thread(target=switch)
    try:
        lqcd.dslash_form(lqcd.DSLASH_PREFETCH)
        single = {solve()}
        lqcd.dslash_form(lqcd.DSLASH_PACKED)
        for block in tables:
            lqcd.autotune_load(tables[block])
            single.add(solve())
        assert all(rc == lqcd.OK for rc, _, _ in single)
        t.start()
        got = [solve() for _ in range(12)]
    finally:
        stop.set()
        if t.is_alive():
            t.join()
        lqcd.dslash_form(form)
        lqcd.autotune_clear()
    assert [rc for rc, _, _ in got] == [lqcd.OK] * len(got)
    assert all(g in single for g in got)


@pytest.mark.parametrize("block", [64, 256])
def test_solve_at_tuned_block_sizes(tmp_path, block):
    """alpha is formed from as many partials as the tuned hop stores: the solve
    takes the iterations of the default block size (another order of the sums,
    so one more or less) to the same solution"""
    U = lqcd.gauge_field(DIMS)
    lqcd.gauge_start(U, 5, 0.2)
    b = lqcd.spinor_field(DIMS, 0)
    lqcd.eta_refresh(b, 6, 0)
    Us = lqcd.gauge_field(DIMS, lqcd.F16N).copy_from(U)
    prm = lqcd.cg_params(tol=1e-10, maxiter=1000, sloppy=lqcd.F16N, delta=0.05)
    got = []
    try:
        for bs in (128, block):
            (tmp_path / "t.txt").write_text("dslash_f16n {} {} {} {} {} 1.0 1\n".format(*DIMS, bs))
            lqcd.autotune_load(tmp_path / "t.txt")
            x = lqcd.spinor_field(DIMS, 0)
            rc, info = lqcd.cg_solve(x, U, b, 0.15, prm, U_sloppy=Us)
            assert rc == lqcd.OK and info.true_rel_res <= 1e-10
            got.append((info.iters, x.download()))
    finally:
        lqcd.autotune_clear()
    assert abs(got[0][0] - got[1][0]) <= 1
    # |dx| / |x| <= 2e-10 times the condition number, which some 40 iterations bound by 500
    assert np.linalg.norm(got[0][1] - got[1][1]) <= 1e-7 * np.linalg.norm(got[0][1])
