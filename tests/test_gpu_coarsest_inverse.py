"""The dense inverse of the coarsest matrix and the Galerkin rows that do not fit
a warp's shared memory.

Block Gauss-Jordan at the edges of its 32-row blocks, through a two-level
hierarchy whose coarsest level has exactly n rows: a block-diagonal fine
matrix of n tightly coupled pairs gives one aggregate per pair, so the coarse
matrix is known, and a single-level handle applies the inverse itself.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_2210_16660_gb300 import binding as B  # noqa: E402
from paper_2210_16660_gb300 import workloads as W  # noqa: E402


def _csr(M):
    n = M.shape[0]
    r, c = np.nonzero(M)
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(r, minlength=n), out=rp[1:])
    return W.CSR(n, rp, c.astype(np.int32), np.ascontiguousarray(M[r, c]))


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 127, 160, 200, 513])
def test_single_level_solve_is_the_inverse(n):
    rng = np.random.default_rng(n)
    # a random SPD matrix of condition about 1e4, exactly symmetric
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    M = (q * np.logspace(0, 4, n)) @ q.T
    M = 0.5 * (M + M.T)
    amg = B.AMG.from_csr(_csr(M), mode="pcg64", coarse_max=n)
    assert len(amg.info()) == 1
    b = rng.standard_normal(n)
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    r = amg.solve(torch.from_numpy(b).cuda(), x, rtol=1e-9)
    # Gauss-Jordan on an SPD matrix: forward error within c n u cond, so one
    # or two iterations meet rtol
    assert r.status == 0 and r.iters <= 2
    assert np.linalg.norm(M @ x.cpu().numpy() - b) <= 1e-9 * np.linalg.norm(b)


def test_indefinite_coarsest_matrix_is_refused():
    M = np.diag(np.full(40, 2.0))
    M[36, 37] = M[37, 36] = -3.0      # a pivot in the second block turns negative
    with pytest.raises(B.AmgError) as e:
        B.AMG.from_csr(_csr(M), coarse_max=40)
    assert e.value.status == B.ERR_BREAKDOWN


@pytest.mark.parametrize("bw", [20, 31, 32, 40, 70])
def test_galerkin_rows_up_to_and_past_the_shared_capacity(bw):
    """Band matrices whose coarse rows have 2 (2 bw + 1) terms: below, at and
    above 128. Hierarchy bit for bit the oracle's."""
    n = 400
    rng = np.random.default_rng(bw)
    M = np.zeros((n, n))
    for d in range(1, bw + 1):
        v = -rng.uniform(0.1, 1.0, n - d)
        M += np.diag(v, d) + np.diag(v, -d)
    M += np.diag(np.abs(M).sum(1) + 0.1)
    A = _csr(M)
    amg = B.AMG.from_csr(A, coarse_max=60, n_pass=2)
    h_or = O.Hierarchy(A, coarse_max=60, n_pass=2)
    assert len(amg.info()) == h_or.nlevels > 1
    for l in range(h_or.nlevels):
        rp, ci, v = amg.level_csr(l)
        lv = h_or.level(l)
        assert np.array_equal(rp, lv["row_ptr"]) and np.array_equal(ci, lv["col"])
        assert np.array_equal(v.view(np.int64), lv["val"].view(np.int64))
