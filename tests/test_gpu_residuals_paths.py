"""The allocation-free residuals on both of their paths (one cluster up to m n =
2^19, three launches above) at the edges of their lanes, blocks and ranges,
against the oracle's residual function.

Tolerance: every output is a quotient of sums of at most n + nnz positive terms
or of their roots (the point is far from feasible, so no residual cancels), each
sum off by at most its number of terms times eps; the two objectives are sums of
signed terms, off by that times the sum of their magnitudes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi  # noqa: E402
from oracle import kkt  # noqa: E402
import scipy.sparse as sp  # noqa: E402

EPS = 2.0 ** -52


@pytest.mark.parametrize("cone", [0, 2, 9, 64])
@pytest.mark.parametrize("m,n,density", [(1, 1, 1.0), (3, 70, 0.5), (31, 33, 1.0), (200, 500, 0.05),
                                         (512, 1024, 0.01), (512, 1025, 0.01), (4000, 9000, 0.002),
                                         (40_000, 3000, 0.002), (700, 1500, 1.0)])
def test_against_the_oracle(m, n, density, cone):
    rng = np.random.default_rng(1000 * m + n + cone)
    A = sp.random(m, n, density=density, format="csr", random_state=rng)
    A.data = rng.standard_normal(A.nnz)
    A.sort_indices()
    dims = np.full(n // (2 * cone), cone, np.int64) if cone else np.zeros(0, np.int64)
    n_orth = n - int(dims.sum())
    b, y = rng.standard_normal(m), rng.standard_normal(m)
    c, x, z = (rng.standard_normal(n) for _ in range(3))
    off = n_orth + np.concatenate([[0], np.cumsum(dims)])
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b, c, x, y, z,
                     off.astype(np.int32))]
    if dev[1].numel() == 0:
        dev[1], dev[2] = (torch.zeros(1, dtype=t.dtype, device="cuda") for t in dev[1:3])
    out = torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")
    ref = kkt.residuals(A, b, c, x, y, z, n_orth, dims)
    terms = 4 * (n + m + A.nnz)
    for _ in range(2):                                   # the second call finds used scratch
        rc = capi.acs_kkt_residuals_noalloc(m, n, *[t.data_ptr() for t in dev[:8]], n_orth, len(dims),
                                            dev[8].data_ptr(), out.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        assert rc == capi.SOLVED
        got = out.cpu().numpy()
        for k, key in enumerate(("r_p", "r_d", "r_cone")):
            v = got[(0, 1, 3)[k]]
            assert abs(v - ref[key]) <= terms * EPS * max(ref[key], EPS), (key, v, ref[key])
        for v, want, mag in ((got[4], ref["obj_p"], np.abs(c * x).sum()), (got[5], ref["obj_d"], np.abs(b * y).sum())):
            assert abs(v - want) <= terms * EPS * mag
        gap = abs(got[4] - got[5]) / (1.0 + abs(got[4]) + abs(got[5]))
        assert abs(got[2] - gap) <= 8 * EPS
