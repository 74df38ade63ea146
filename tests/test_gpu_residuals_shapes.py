"""The allocation-free residuals of tall, wide and many-coned problems: against the
oracle's residual function, and with short cones no dearer than their entries.

Tolerance: as for the residuals' other tests, every output is a quotient of sums of
at most n + nnz positive terms or of their roots, each off by at most its number of
terms times eps; the two objectives by that times the sum of their magnitudes.
Times: the smallest of several, as the ratio of two calls, bounded by about one and a
half times what it should be.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi  # noqa: E402
from oracle import kkt  # noqa: E402
import scipy.sparse as sp  # noqa: E402

EPS = 2.0 ** -52


class Case:
    def __init__(self, m, n, per_row, dims):
        rng = np.random.default_rng(m + n + len(dims))
        step = n // per_row
        cols = np.arange(per_row) * step + rng.integers(0, step, (m, per_row))
        self.m, self.n, self.dims = m, n, np.asarray(dims, np.int64)
        self.A = sp.csr_matrix((rng.standard_normal(m * per_row), cols.reshape(-1).astype(np.int32),
                                np.arange(0, m * per_row + 1, per_row, dtype=np.int32)), shape=(m, n))
        self.n_orth = n - int(self.dims.sum())
        self.b, self.y = rng.standard_normal(m), rng.standard_normal(m)
        self.c, self.x, self.z = (rng.standard_normal(n) for _ in range(3))
        off = (self.n_orth + np.concatenate([[0], np.cumsum(self.dims)])).astype(np.int32)
        self.dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
                    for a in (self.A.indptr, self.A.indices, self.A.data, self.b, self.c, self.x, self.y, self.z, off)]
        self.out = torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")

    def call(self):
        rc = capi.acs_kkt_residuals_noalloc(self.m, self.n, *[t.data_ptr() for t in self.dev[:8]], self.n_orth,
                                            len(self.dims), self.dev[8].data_ptr(), self.out.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        assert rc == capi.SOLVED

    def us(self):
        best = np.inf
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(10):
                self.call()
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1) * 100.0)
        return best


@pytest.mark.parametrize("m,n,per_row", [(1, 524_288, 524_288), (3, 170_000, 170_000), (50_000, 10, 3),
                                         (524_288, 1, 1), (2048, 256, 10), (2049, 256, 10), (64, 16_384, 10),
                                         (63, 16_385, 10), (1024, 1024, 1024), (1, 1 << 20, 10), (9728, 77_824, 9),
                                         (9729, 77_825, 9)])
def test_shapes(m, n, per_row):
    _check(Case(m, n, per_row, []))


@pytest.mark.parametrize("m,n", [(1, 524_286), (1, 16_382), (3, 8190), (64, 16_380)])
def test_wide_with_cones(m, n):
    """Lanes of one warp with different numbers of coordinates, all of them in cones of 3."""
    _check(Case(m, n, 10, [3] * (n // 3)))


# cones of a mean length up to 9 are added up eight to a group of eight lanes, longer ones one to a group
CONES = {"one": [7], "seven": [2, 3, 8, 9, 10, 5, 4], "eight": [9] * 8, "thirty-three": [3] * 33,
         "a long one among short ones": [2] * 40 + [150] + [3] * 40, "of 10": [10] * 31, "of 64": [64] * 5,
         "many": [2] * 400}


@pytest.mark.parametrize("cones", sorted(CONES))
@pytest.mark.parametrize("m", [40, 2600])
@pytest.mark.parametrize("n_orth", [0, 13])
def test_cones(cones, m, n_orth):
    n = n_orth + sum(CONES[cones])
    _check(Case(m, n, min(n, 4), CONES[cones]))


def _check(P):
    ref = kkt.residuals(P.A, P.b, P.c, P.x, P.y, P.z, P.n_orth, P.dims)
    terms = 4 * (P.n + P.m + P.A.nnz)
    for _ in range(2):                                   # the second call finds used scratch
        P.call()
        got = P.out.cpu().numpy()
        for k, key in enumerate(("r_p", "r_d", "r_cone")):
            assert abs(got[(0, 1, 3)[k]] - ref[key]) <= terms * EPS * max(ref[key], EPS), key
        for v, want, mag in ((got[4], ref["obj_p"], np.abs(P.c * P.x).sum()),
                             (got[5], ref["obj_d"], np.abs(P.b * P.y).sum())):
            assert abs(v - want) <= terms * EPS * mag


def test_short_cones_cost_little():
    """5e5 cones of 2 beside 1e7 nonzeros."""
    assert Case(200_000, 1_000_000, 50, [2] * 500_000).us() <= 2.0 * Case(200_000, 1_000_000, 50, []).us()
