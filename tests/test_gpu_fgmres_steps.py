"""Arnoldi steps of the outer FGMRES at the sizes where their kernels can go wrong:
restart lengths around the groups of eight columns and at the largest, steps across
a restart, systems of less than a warp, one level, and with and without the captured
step."""
import numpy as np
import pytest

from paper_1403_1649_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle
    from paper_1403_1649_gb300 import amg, build
    build.build()
    oracle.build()
    return amg, oracle


@pytest.mark.parametrize("restart", [1, 7, 8, 9, 25, 32])
@pytest.mark.parametrize("graph", [0, 1])
def test_steps_match_the_oracle_across_a_restart(env, restart, graph):
    amg, oracle = env
    A = P.convdiff2d(43, 11, pe=3.0)
    b = P.rhs_uniform(A.n, 5)
    # a weak smoother, so that no step of the count reaches rounding
    kw = dict(alpha=0.25, seed=3, symmetric=0, outer=1, restart=restart, omega_mode=1, omega=0.05)
    steps = restart + 3
    xg, ig = amg.Hierarchy(A, use_graph=graph, max_iter=steps, **kw).solve(
        b, tol=0.0, allow=(amg.AMG_OK, amg.AMG_ERR_NOT_CONVERGED))
    xo, io = oracle.Hierarchy(A, **kw).solve(b, tol=0.0, max_iter=steps)
    assert ig["iters"] == io["iters"] == steps
    assert np.allclose(ig["hist"], io["hist"], rtol=1e-6, atol=1e-12)
    assert np.linalg.norm(xg - xo) <= 1e-8 * np.linalg.norm(xo)


@pytest.mark.parametrize("m,coarse,prec", [(3, 64, 0), (7, 64, 1), (16, 16, 0), (131, 64, 0), (131, 64, 1), (131, 64, 2)])
def test_solve_reaches_the_tolerance(env, m, coarse, prec):
    amg, _ = env
    A = P.convdiff2d(m, 2, pe=2.0)
    b = P.rhs_uniform(A.n, 9)
    h = amg.Hierarchy(A, alpha=0.25, seed=1, symmetric=0, outer=1, restart=10, coarse_max=coarse, precision=prec,
                      max_iter=300)
    for _ in range(2):  # the captured step serves the second solve too
        x, info = h.solve(b, tol=1e-10)
        assert info["status"] == amg.AMG_OK
        assert np.linalg.norm(b - A.matvec(x)) <= 1e-10 * np.linalg.norm(b) * (1 + 1e-6)
    x, info = h.solve(np.zeros(A.n), tol=1e-10)
    assert info["iters"] == 0 and not x.any()
