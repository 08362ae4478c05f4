"""Tuning times the packed hopping term whatever form is set, and leaves the
process-wide setting alone while it does: another thread's launches keep theirs."""
import threading

import pytest

from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu


def test_autotune_leaves_the_form_alone():
    form = lqcd.dslash_form(lqcd.DSLASH_PREFETCH)
    seen, done = set(), threading.Event()

    def watch():
        while not done.is_set():
            seen.add(lqcd.dslash_form())

    t = threading.Thread(target=watch)
    t.start()
    try:
        lqcd.autotune((16, 16, 16, 16))
    finally:
        done.set()
        t.join()
        lqcd.dslash_form(form)
        lqcd.autotune_clear()
    assert seen == {lqcd.DSLASH_PREFETCH}
