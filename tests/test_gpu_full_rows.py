"""Matrices whose rows hold every column, at the edges of the assembly's 32 x 32 tiles
and 16-entry slabs and of the dense products' eight entries a lane, in every launch
that takes them: single problems, teams of 256, 512 and 1024 threads, served requests, the
FP32 and BF16 values of the CG.  Iterates equal the oracle's, which projects exactly.

Tolerance with the cached operator: an iteration solves with M = A A' once; a
backward-stable solve of an m x m system is off by about m eps cond(M), and k iterations of
a nonexpansive map add up to k times that (relative to the iterate).  With CG the bar of
the FP32 iterates, 1e-4.
"""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402
from oracle import alg  # noqa: E402

ITERS = 20
SIZES = (15, 16, 17, 31, 32, 33, 65, 160, 257)
MAPPINGS = [(256, 1), (256, 2), (256, 8), (512, 1), (512, 4), (1024, 1), (1024, 2)]


def _full_lp(m, n=None):
    n = n or 2 * m + 1
    rng = np.random.default_rng(4000 + m)
    A = sp.csr_matrix(rng.standard_normal((m, n)))
    return I.planted_lp(A.indptr, A.indices, A.data, m, n, seed=m)


def _reference(inst, A=None, b=None, t=9.2, L=alg.LP_SCHEDULE):
    A, b = inst.to_scipy() if A is None else A, inst.b if b is None else b
    r = alg.algorithm2(A, b, inst.c, inst.n_orth, inst.soc_dims, t=t, L=L, max_iter=ITERS, tol=0.0)
    D = A.toarray()
    return r.x, r.z, max(ITERS * A.shape[0] * 2.0 ** -52 * np.linalg.cond(D @ D.T), 1e-14)


def _close(got, ref, tol=None):
    rc, x, y, z, iters, res = got[:6]
    assert rc == capi.MAX_ITER and iters == ITERS
    for v, want in ((x, ref[0]), (z, ref[1])):
        assert np.linalg.norm(v - want) <= (tol or ref[2]) * np.linalg.norm(want)


@pytest.mark.parametrize("precision", [capi.PREC_MIXED, capi.PREC_FP64])
@pytest.mark.parametrize("m", SIZES + (511, 1025))       # the last two on the whole grid
def test_single(m, precision):
    inst = _full_lp(m, m + 200 if m > 500 else None)
    with capi.Solver(inst, projection=capi.PROJ_DENSE, precision=precision) as s:
        s.solve(tol=0.0, max_iter=ITERS)
        _close(s.get(), _reference(inst))


@pytest.mark.parametrize("mapping", MAPPINGS)
def test_teams(mapping):
    members = [_full_lp(m) for m in SIZES]
    with capi.Batch(members, mapping=mapping, share=None, projection=capi.PROJ_DENSE) as b:
        b.solve(tol=0.0, max_iter=ITERS)
        for i, inst in enumerate(members):
            _close(b.get(i), _reference(inst))


@pytest.mark.parametrize("dependent", [3, 20, 39, 200, 256])
def test_dependent_row(dependent):
    """A repeated row in the first, a middle and the last (partial) block of 16 columns
    is dropped: the iterates are those of the problem without it."""
    m = 40 if dependent < 40 else 257
    inst = _full_lp(m)
    D = inst.to_scipy().toarray()
    D[dependent] = -2.0 * D[dependent - 2]
    inst.val, inst.b = D.reshape(-1).copy(), inst.b.copy()
    inst.b[dependent] = -2.0 * inst.b[dependent - 2]
    keep = np.arange(m) != dependent
    ref = _reference(inst, sp.csr_matrix(D[keep]), inst.b[keep])
    with capi.Solver(inst, projection=capi.PROJ_DENSE) as s:
        s.solve(tol=0.0, max_iter=ITERS)
        _close(s.get(), ref)
    for mapping in ((256, 2), (512, 1)):
        with capi.Batch([inst], mapping=mapping, share=None, projection=capi.PROJ_DENSE) as b:
            b.solve(tol=0.0, max_iter=ITERS)
            _close(b.get(0), ref)


@pytest.mark.parametrize("threads", [256, 512])
def test_served(threads):
    requests = [I.dense_socp(n, 10, seed=n) for n in (20, 50, 160, 330)] + [_full_lp(m) for m in (15, 33, 160)]
    with capi.Server(threads_per_cta=threads) as S:
        ids = [S.submit(r, tol=0.0, max_iter=ITERS) for r in requests]
        for r, i in zip(requests, ids):
            assert S.wait(i, timeout_s=60.0) != capi.ERR_DEVICE_TIMEOUT
            _close(S.result(i), _reference(r, t=1.7, L=alg.SOCP_SCHEDULE) if len(r.soc_dims) else _reference(r))


CG = dict(projection=capi.PROJ_CG, cg_eta=1e-9, cg_tol=0.0)


@pytest.mark.parametrize("m", [15, 32, 65, 160])
def test_cg_values(m):
    """The CG's passes over full rows, FP32 values, one problem and teams."""
    inst = _full_lp(m)
    ref = _reference(inst)
    with capi.Solver(inst, **CG) as s:
        s.solve(tol=0.0, max_iter=ITERS)
        _close(s.get(), ref, 1e-4)
    for mapping in ((256, 1), (512, 2)):
        with capi.Batch([inst], mapping=mapping, share=None, **CG) as b:
            b.solve(tol=0.0, max_iter=ITERS)
            _close(b.get(0), ref, 1e-4)


@pytest.mark.parametrize("m", [15, 32, 65, 160])
def test_bf16_values(m):
    """BF16 values on full rows: the refinement-step model's iterates."""
    import refinement_model as RM
    inst = _full_lp(m)
    A = inst.to_scipy()
    ref = RM.refined_iterates(A, inst.b, inst.c, inst.n, [], iters=ITERS, correction_values=RM.bf16_round(A.data))[-1]
    with capi.Solver(inst, a_storage=capi.STORE_BF16, **CG) as s:
        s.solve(tol=0.0, max_iter=ITERS)
        x = s.get()[1]
    assert np.linalg.norm(x - ref) <= 1e-4 * np.linalg.norm(ref)
    with capi.Batch([inst], mapping=(256, 2), share=None, a_storage=capi.STORE_BF16, **CG) as b:
        b.solve(tol=0.0, max_iter=ITERS)
        x = b.get(0)[1]
    assert np.linalg.norm(x - ref) <= 1e-4 * np.linalg.norm(ref)
