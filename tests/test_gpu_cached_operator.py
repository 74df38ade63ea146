"""The cached projection operator at the edges of its blocks (16 columns) and
tiles (32 x 32), in the single-problem launch and in teams of one and two
CTAs of every size: iterates equal the oracle's, which projects exactly.

Tolerance: an iteration solves with M = A A' once; a backward-stable solve of
an m x m system is off by about m eps cond(M), and k iterations of a
nonexpansive map add up to k times that (relative to the iterate).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402
from oracle import alg  # noqa: E402

ITERS = 20
SIZES = (1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 100, 257, 511)


def _instance(m):
    return I.bernoulli_lp(7000 + m, m, int(2.5 * m) + 3, density=min(1.0, 0.02 + 3.0 / m))


def _reference(inst):
    r = alg.algorithm2(inst.to_scipy(), inst.b, inst.c, inst.n, [], L=alg.LP_SCHEDULE, max_iter=ITERS, tol=0.0)
    A = inst.to_scipy().toarray()
    return r.x, r.z, ITERS * inst.m * 2.0 ** -52 * np.linalg.cond(A @ A.T)


def _close(x, z, ref):
    xr, zr, tol = ref
    tol = max(tol, 1e-14)
    assert np.linalg.norm(x - xr) <= tol * np.linalg.norm(xr)
    assert np.linalg.norm(z - zr) <= tol * np.linalg.norm(zr)


@pytest.mark.parametrize("m", SIZES + (1000, 1025))
def test_single(m):
    inst = _instance(m)
    with capi.Solver(inst, projection=capi.PROJ_DENSE) as s:
        for _ in range(2):                               # fresh scratch, then used scratch
            s.solve(tol=0.0, max_iter=ITERS)
            rc, x, y, z, iters, res = s.get()
            assert rc == capi.MAX_ITER and iters == ITERS
            _close(x, z, _reference(inst))


@pytest.mark.parametrize("mapping", [(256, 1), (256, 2), (512, 1), (512, 4), (1024, 1), (1024, 2)])
def test_teams(mapping):
    members = [_instance(m) for m in SIZES]
    refs = [_reference(i) for i in members]
    with capi.Batch(members, mapping=mapping, share=None, projection=capi.PROJ_DENSE) as b:
        b.solve(tol=0.0, max_iter=ITERS)
        for i, ref in enumerate(refs):
            rc, x, y, z, iters, res = b.get(i)
            assert rc == capi.MAX_ITER and iters == ITERS
            _close(x, z, ref)
