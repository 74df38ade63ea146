"""Wide problems on either side of the one-cluster launch's limit of 16384 coordinates,
with lanes of one warp that have different numbers of them: the launch, and iterates
equal to the oracle's, which projects exactly.

Tolerance: as for the cached operator, k iterations of a nonexpansive map, each with a
solve off by about m eps cond(M); sums over n coordinates add n eps.
"""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402
from oracle import alg  # noqa: E402

ITERS = 12


@pytest.mark.parametrize("n,small", [(8193, True), (12_301, True), (16_383, True), (16_384, True), (16_385, False),
                                     (40_003, False)])
def test_wide(n, small, m=24):
    rng = np.random.default_rng(n)
    A = sp.csr_matrix((rng.standard_normal(2 * n), (np.concatenate([np.arange(n) % m, (np.arange(n) * 7 + 5) % m]),
                                                    np.concatenate([np.arange(n)] * 2))), shape=(m, n))
    A.sum_duplicates()
    inst = I.planted_lp(A.indptr, A.indices, A.data, m, n, seed=n)
    ref = alg.algorithm2(A, inst.b, inst.c, n, [], L=alg.LP_SCHEDULE, max_iter=ITERS, tol=0.0)
    tol = ITERS * (m * np.linalg.cond((A @ A.T).toarray()) + n) * 2.0 ** -52
    with capi.Solver(inst, projection=capi.PROJ_DENSE) as s:
        assert (capi.acs_problem_info(s.h)["threads"] == 512) == small
        s.solve(tol=0.0, max_iter=ITERS)
        rc, x, y, z, iters, res = s.get()
    assert rc == capi.MAX_ITER and iters == ITERS
    assert np.linalg.norm(x - ref.x) <= tol * np.linalg.norm(ref.x)
    assert np.linalg.norm(z - ref.z) <= tol * np.linalg.norm(ref.z)
