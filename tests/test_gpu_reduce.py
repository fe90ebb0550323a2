"""Sums over threads, blocks and partials on the integer pipe (csrc/reduce.cuh).

The solve's scalars (r.z, z.q, p.q, ||r||^2) scale exactly with powers of two
as long as nothing leaves the normal range, so a system scaled by 2^k must
give the same iterates, bit for bit, as the unscaled one: the alignment to the
largest exponent, the headroom and the conversion back are then right at
every magnitude. Sizes cover one block, ragged warps and several blocks.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2210_16660_gb300 import binding as B  # noqa: E402
from paper_2210_16660_gb300 import workloads as W  # noqa: E402


def _solve(amg, b, x0, **kw):
    x = x0.clone()
    return amg.solve(b, x, rtol=1e-8, **kw), x


@pytest.mark.parametrize("N", [5, 7, 13, 33, 45])
@pytest.mark.parametrize("mode,ks", [("pcg64", (-480, -300, 300, 480)), ("fcg32", (-40, 40))])
def test_power_of_two_scaling_is_exact(N, mode, ks):
    prob = W.make_problem(N, 1.04, seed=11)
    amg = B.AMG.from_csr(prob.A, mode=mode)
    # magnitudes spread over 2^+-20, so partials differ in exponent and sign
    x0 = torch.from_numpy(W.normals(5, prob.A.n) * 2.0 ** (np.arange(prob.A.n) % 41 - 20.0)).cuda()
    b = torch.from_numpy(prob.b).cuda()
    r0, y0 = _solve(amg, b, x0)
    assert r0.status == 0
    # the first residual against the host's own sums: row sums of up to 27
    # products and a sum over n squares, each rounded, so within (27 + 2) u
    # of sum |a||x| + |b| per row
    A, xs = prob.A, x0.cpu().numpy()
    res = prob.b - W.spmv(A, xs)
    absrow = W.spmv(W.CSR(A.n, A.row_ptr, A.col, np.abs(A.val)), np.abs(xs)) + np.abs(prob.b)
    bound = 2.0 * 29 * 2.0 ** -53 * np.linalg.norm(absrow) / np.linalg.norm(prob.b)
    assert abs(r0.hist[0] - np.linalg.norm(res) / np.linalg.norm(prob.b)) <= bound + 4 * 2.0 ** -53 * r0.hist[0]
    for k in ks:
        s = 2.0 ** k
        r, y = _solve(amg, b * s, x0 * s)
        assert r.status == 0 and r.iters == r0.iters
        assert np.array_equal(r.hist, r0.hist)
        assert torch.equal(y, y0 * s)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_sums_end_the_solve(bad):
    prob = W.make_problem(13, 1.04, seed=12)
    amg = B.AMG.from_csr(prob.A, mode="pcg64")
    b = torch.from_numpy(prob.b).cuda()
    b[prob.A.n - 1] = bad
    r, _ = _solve(amg, b, torch.zeros_like(b))
    assert r.status == B.ERR_NAN


def test_outcomes_do_not_depend_on_when_blocks_start():
    """Branches of a batch delay one another's blocks, so a block may start
    after the one that records an iteration's outcome: every repetition still
    equals the systems' own solves bit for bit."""
    probs = [W.make_problem(N, 1.04, seed=60 + N) for N in (61, 44, 38, 31, 29, 45, 52)]
    amgs = [B.AMG.from_csr(p.A, mode="fcg32") for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    alone = []
    for a, b in zip(amgs, bs):
        r, y = _solve(a, b, torch.zeros_like(b))
        assert r.status == 0
        alone.append((r.iters, y))
    batch = B.Batch(amgs)
    for _ in range(12):
        xs = [torch.zeros_like(b) for b in bs]
        st, it, _ = batch.solve(bs, xs)
        assert st == 0
        for k, (iters, y) in enumerate(alone):
            assert it[k] == iters and torch.equal(xs[k], y), k
    batch.close()
