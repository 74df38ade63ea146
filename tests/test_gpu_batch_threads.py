"""Results of one batch read by two threads at once: every call returns its own
member's, however long the other's copy takes."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402


def _diagonal_lp(m, n):
    """One entry a column, row j mod m."""
    rng = np.random.default_rng(m)
    rows = np.arange(n) % m
    order = np.argsort(rows, kind="stable")
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    return I.planted_lp(row_ptr, order, rng.uniform(0.5, 2.0, n), m, n, seed=n)


def test_two_readers():
    members = [_diagonal_lp(50_000, 150_000), _diagonal_lp(40, 100)]
    with capi.Batch(members, share=None) as b:
        b.solve(tol=0.0, max_iter=3)
        want = [b.get(i) for i in range(2)]
        wrong, stop = [0, 0], threading.Event()

        def read(i, times):
            while times > 0 and not stop.is_set():
                times -= i == 0
                got = b.get(i)
                wrong[i] += not (got[0] == want[i][0] and all(np.array_equal(got[k], want[i][k]) for k in (1, 2, 3)))
            stop.set()

        readers = [threading.Thread(target=read, args=a) for a in ((0, 200), (1, 1))]
        for t in readers:
            t.start()
        for t in readers:
            t.join()
    assert wrong == [0, 0]
