"""Calls on a batch hierarchy beside amg_solve_batch, before and after it: products
and preconditioner applications do not depend on which systems the last solve
stopped."""
import numpy as np
import pytest

from paper_1403_1649_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_1649_gb300 import amg, build
    build.build()
    amg.lib()
    return torch, amg


UNEVEN = [20, 33, 47, 12, 60, 8, 29]


def batch(sides):
    mats = [P.varcoef2d(m, 40 + q) for q, m in enumerate(sides)]
    return mats, np.concatenate([P.rhs_uniform(A.n, 60 + q) for q, A in enumerate(mats)])


class Batch:
    def __init__(self, amg, mats, **params):
        self.amg, self.n = amg, sum(A.n for A in mats)
        self.h = amg.amg_setup_batch(mats, amg.amg_default_params(alpha=0.25, seed=1, **params))
        self.levels = amg.amg_hierarchy_info(self.h)

    def __del__(self):
        if getattr(self, "h", None):
            self.amg.amg_free(self.h)

    def precond(self, b):
        x = np.zeros(self.n)
        self.amg.amg_precond(self.h, b, x)
        return x


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("sides", [UNEVEN, [45], [24, 24]])
def test_product_and_preconditioner_after_a_solve(env, prec, sides):
    """After a solve in which the systems stopped one by one (or all together), every
    level's product and the preconditioner are those of a hierarchy that has not
    solved; the FP64 product is that of the level matrix."""
    torch, amg = env
    mats, b = batch(sides)
    solved, fresh = Batch(amg, mats, precision=prec), Batch(amg, mats, precision=prec)
    rc, it, rel = amg.amg_solve_batch(solved.h, b, np.zeros_like(b), 1e-8, len(mats))
    assert rc == amg.AMG_OK and (rel <= 1e-8).all()
    for k, lv in enumerate(solved.levels):
        x = P.rhs_uniform(lv["n"], 5 + k).astype(np.float64 if prec == 0 else np.float32)
        y = []
        for g in (solved, fresh):
            xd = torch.from_numpy(x).cuda()
            yd = torch.full_like(xd, float("nan"))
            amg.amg_spmv(g.h, k, xd, yd)
            torch.cuda.synchronize()
            y.append(yd.cpu().numpy())
        assert np.array_equal(y[0], y[1]), k
        if prec == 0:
            L = amg.amg_export_level(solved.h, k)
            Ak = P.CSR(L["n"], L["rowptr"], L["col"], L["val"])
            mag = P.CSR(Ak.n, Ak.rowptr, Ak.col, np.abs(Ak.val)).matvec(np.abs(x))
            w = np.diff(Ak.rowptr) + 4.0
            assert (np.abs(y[0] - Ak.matvec(x)) <= 2 * w * 2.0 ** -53 * mag).all(), k
    assert np.array_equal(solved.precond(b), fresh.precond(b))


@pytest.mark.parametrize("prec", [0, 1])
def test_solve_after_a_system_ran_into_infinities(env, prec):
    """A right-hand side outside the preconditioner's range ends one system of a batch
    with a failure code; the next solve on the same hierarchy, with ordinary data, is
    that of a fresh one."""
    _, amg = env
    mats, b = batch(UNEVEN)
    used, fresh = Batch(amg, mats, precision=prec), Batch(amg, mats, precision=prec)
    n0, n1 = mats[0].n, mats[0].n + mats[1].n
    bad = b.copy()
    bad[n0:n1] *= 1e60 if prec else 1e152  # squares overflow on the way, the norm does not
    rc, it, rel = amg.amg_solve_batch(used.h, bad, np.zeros_like(b), 1e-8, len(mats),
                                      allow=(amg.AMG_OK, amg.AMG_ERR_BREAKDOWN, amg.AMG_ERR_NAN))
    x = [np.zeros_like(b), np.zeros_like(b)]
    for g, xs in ((used, x[0]), (fresh, x[1])):
        rc, it, rel = amg.amg_solve_batch(g.h, b, xs, 1e-8, len(mats), allow=(amg.AMG_OK, amg.AMG_ERR_BREAKDOWN,
                                                                             amg.AMG_ERR_NAN))
        assert rc == amg.AMG_OK and (rel <= 1e-8).all()
    assert np.array_equal(*x)
