"""Transfers inside the small levels' sweeps, and the small levels as one matrix.

The down sweep that restricts in the same launch (member order) and the
kernels that prolong the x they form give the bits of the separate launches
(PCGAMG_TAIL=0): checked for aggregates of 2 to 64 rows (slots of 2 to 32, and
past a warp the separate launches), ragged sizes and both column widths. The
explicit matrix of the small levels (left out by PCGAMG_OP=0) is the same
operator as the levels one by one, up to rounding.
"""
import ctypes as C
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2210_16660_gb300 import binding as B  # noqa: E402
from paper_2210_16660_gb300 import workloads as W  # noqa: E402
from test_gpu_parity import direct_level  # noqa: E402


def _amg(A, env=(), **kw):
    old = {k: os.environ.get(k) for k, _ in env}
    os.environ.update(dict(env))
    try:
        return B.AMG.from_csr(A, **kw)
    finally:
        for k, v in old.items():
            if v is None:
                del os.environ[k]
            else:
                os.environ[k] = v


def _solve(amg, b):
    x = torch.zeros_like(b)
    return amg.solve(b, x, rtol=1e-8), x


@pytest.mark.parametrize("mode", ["pcg64", "fcg32"])
@pytest.mark.parametrize("N,npass,cmax,env", [
    (9, 1, 10, ()), (14, 2, 20, ()), (24, 3, 30, (("PCGAMG_COL16", "0"),)), (33, 4, 20, (("PCGAMG_UNIFORM", "0"),)),
    (24, 5, 5, ()), (24, 6, 5, ()), (41, 2, 200, ()), (33, 1, 3000, ())])
def test_fused_transfers_give_the_bits_of_separate_launches(N, npass, cmax, env, mode):
    prob = W.make_problem(N, 1.04, seed=3)
    b = torch.from_numpy(prob.b).cuda()
    kw = dict(mode=mode, n_pass=npass, coarse_max=cmax)
    r1, x1 = _solve(_amg(prob.A, env, **kw), b)
    r2, x2 = _solve(_amg(prob.A, tuple(env) + (("PCGAMG_TAIL", "0"),), **kw), b)
    assert r1.status == r2.status == 0 and r1.iters == r2.iters
    assert np.array_equal(r1.hist, r2.hist) and torch.equal(x1, x2)


class Bytes:
    """An allocator that counts the library's bytes and refuses past `limit`."""

    def __enter__(self):
        self.live, self.now, self.peak, self.limit = {}, 0, 0, None

        def alloc(n, stream, ctx):
            if self.limit is not None and self.now + n > self.limit:
                return None
            p = torch.cuda.caching_allocator_alloc(int(n), torch.cuda.current_device(), stream or 0)
            self.live[p] = n
            self.now += n
            self.peak = max(self.peak, self.now)
            return p

        def free(p, stream, ctx):
            self.now -= self.live.pop(p)
            torch.cuda.caching_allocator_delete(p)

        self.refs = (B.ALLOC_FN(alloc), B.FREE_FN(free))
        assert B.load().amg_set_allocator(C.cast(self.refs[0], C.c_void_p), C.cast(self.refs[1], C.c_void_p), None) == 0
        return self

    def __exit__(self, *a):
        B.load().amg_set_allocator(None, None, None)


def _up(n, to):
    return -(-n // to) * to


@pytest.mark.parametrize("N,npass", [(24, 2), (14, 3)])
def test_member_order_is_left_out_of_a_budget_without_room(N, npass):
    """With int32 columns kept nothing is given back for the member order or the
    explicit matrix: a budget of the rest is enough for the hierarchy."""
    prob = W.make_problem(N, 1.04, seed=3)
    b = torch.from_numpy(prob.b).cuda()
    env = (("PCGAMG_COL16", "0"), ("PCGAMG_TAIL", "0"))
    with Bytes() as mem:
        a1 = _amg(prob.A, env, n_pass=npass)
        rows = [n for n, _ in a1.info()]
        extra = 0
        for l, n in enumerate(rows[:-1]):
            agg = a1.level_agg(l, -1)[0]
            cnt = np.bincount(agg[agg >= 0], minlength=rows[l + 1])
            slot = 1 << int(cnt.max() - 1).bit_length()
            extra += _up(4 * (_up(slot * rows[l + 1], 32) + _up(int((agg < 0).sum()), 32)), 256)
            if l > 0 and n <= 1280:
                extra += _up(8 * n * n, 256)
        r1, x1 = _solve(a1, b)
        need = mem.peak - extra
        a1.close()
        a2 = _amg(prob.A, env, n_pass=npass, hbm_budget=need)
        r2, x2 = _solve(a2, b)
        a2.close()
    assert r1.status == r2.status == 0 and abs(r1.iters - r2.iters) <= 1
    assert (x1 - x2).norm().item() <= 1e-6 * x2.norm().item()


@pytest.mark.parametrize("mode", ["pcg64", "fcg32"])
@pytest.mark.parametrize("N,kw,nu,rows", [
    (24, {}, 0, 1), (33, {}, 0, 1), (24, {}, 2, 5), (28, {}, 4, 32), (24, {"smoothed": True, "n_pass": 3}, 0, 1),
    (20, {"coarse_max": 20}, 1, 1)])
def test_small_levels_as_one_matrix(N, kw, nu, rows, mode):
    prob = W.make_problem(N, 1.04, seed=4)
    b = torch.from_numpy(prob.b).cuda()
    A2 = W.rescaled(prob.A, seed=9)
    amgs = [_amg(prob.A, mode=mode, **kw),
            _amg(prob.A, (("PCGAMG_OP", "0"), ("PCGAMG_TAIL", "0")), mode=mode, **kw)]
    L = len(amgs[0].info()) - 1
    assert direct_level(amgs[0], b) < L and direct_level(amgs[1], b) == L
    for step in ("setup", "refresh"):
        out = []
        for a in amgs:
            if step == "refresh":
                a.refresh(A2)
            elif nu:
                a.set_smoother(nu, -(-prob.A.n // rows))
            r, x = _solve(a, b)
            assert r.status == 0, r.message
            out.append((r, x))
        (r1, x1), (r2, x2) = out
        assert abs(r1.iters - r2.iters) <= 1
        # the two V-cycles differ by rounding alone: u = 2^-53 per operation in
        # float64 (2^-24 in float32), a few hundred operations deep, so the
        # residuals of the first iterations agree to 1e-10 (1e-4)
        k = min(5, r1.iters, r2.iters)
        assert np.allclose(r1.hist[:k], r2.hist[:k], rtol=1e-10 if mode == "pcg64" else 1e-4, atol=0)
        assert (x1 - x2).norm().item() <= 1e-6 * x2.norm().item()
    for a in amgs:
        a.close()


@pytest.mark.parametrize("mode", ["pcg64", "fcg32"])
@pytest.mark.parametrize("N,k,env", [(13, 3, ()), (28, 9, (("PCGAMG_UNIFORM", "0"),)), (28, 20, (("PCGAMG_COL16", "0"),)),
                                     (33, 32, ()), (41, 5, ())])
def test_columns_agree_with_single_solves(N, k, env, mode):
    """The coarse levels' multi-column kernels and the explicit operator (whose
    level depends on the column count) against each column solved alone."""
    prob = W.make_problem(N, 1.04, seed=5)
    Bm, _ = W.make_rhs(prob, k, seed=77)
    Bd = torch.from_numpy(np.ascontiguousarray(Bm)).cuda()
    amg = _amg(prob.A, env, mode=mode)
    X = torch.zeros_like(Bd)
    st, it, _, sts, tr = amg.solve_multi(Bd, X, rtol=1e-8)
    assert st == 0 and not sts.any() and (tr <= 1e-8).all()
    for c in (0, k // 2, k - 1):
        r, x = _solve(amg, Bd[:, c].contiguous())
        assert abs(r.iters - int(it[c])) <= 1
        assert (x - X[:, c]).norm().item() <= 1e-6 * x.norm().item()
    amg.close()
