"""Lorentz cones shared by 4, 8, 16 and 32 lanes, at sizes around the lanes'
rounds and mixed with a long one: iterates and residuals equal the oracle's, which
projects exactly.

Tolerance: as for the cached operator, k iterations of a nonexpansive map, each
with a solve off by about m eps cond(M); the cones' own sums add n eps.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402
from oracle import alg, kkt  # noqa: E402

ITERS = 20


@pytest.mark.parametrize("dims,lanes", [([2], 4), ([2, 3, 4, 5, 31, 32, 33, 48], 4), ([49] * 12, 8), ([100] * 9, 16),
                                        ([200] * 7, 32), ([3] * 40 + [300], 8), ([3] * 40 + [600], 16),
                                        ([3] * 40 + [2100], 32), ([2] * 1500, 4)])
@pytest.mark.parametrize("n_orth", [0, 37])
def test_iterates(dims, lanes, n_orth):
    rng = np.random.default_rng(sum(dims) + len(dims) + n_orth)
    n = n_orth + sum(dims)
    m = max(1, min(60, n // 2))
    A = rng.standard_normal((m, n))
    x0, c = rng.standard_normal(n), rng.standard_normal(n)
    nan = np.full(n, np.nan)
    inst = I.Instance(m=m, n=n, row_ptr=np.arange(0, m * n + 1, n, dtype=np.int64),
                      col=np.tile(np.arange(n, dtype=np.int32), m), val=A.reshape(-1), b=A @ x0, c=c, n_orth=n_orth,
                      soc_dims=np.array(dims, np.int32), x_star=nan, y_star=np.full(m, np.nan), s_star=nan)
    ref = alg.algorithm2(inst.to_scipy(), inst.b, inst.c, n_orth, dims, L=alg.LP_SCHEDULE, max_iter=ITERS, tol=0.0)
    tol = ITERS * (m * np.linalg.cond(A @ A.T) + n) * 2.0 ** -52
    with capi.Solver(inst, projection=capi.PROJ_DENSE) as s:
        s.solve(tol=0.0, max_iter=ITERS)
        rc, x, y, z, iters, res = s.get()
    assert rc == capi.MAX_ITER and iters == ITERS
    assert np.linalg.norm(x - ref.x) <= tol * np.linalg.norm(ref.x)
    assert np.linalg.norm(z - ref.z) <= tol * np.linalg.norm(ref.z)
    own = kkt.residuals(inst.to_scipy(), inst.b, inst.c, x, y, z, n_orth, dims)
    assert abs(res[3] - own["r_cone"]) <= n * 2.0 ** -52 * (1.0 + own["r_cone"])
    assert abs(res[4] - own["obj_p"]) <= n * 2.0 ** -52 * np.abs(c * x).sum()
