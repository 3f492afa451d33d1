"""Rows with many weak couplings (a hub joined to hundreds or thousands of grid
points): A P of such rows, the cycle that reads it, and a setup whose time stays
proportional to the row's length."""
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
    amg.lib()
    return amg, oracle


def hub_grid(m, degree, seed):
    """Poisson on an m x m grid; the middle point is also joined to `degree` others by
    couplings of 1e-3, too weak to aggregate over, so that its row of A P meets nearly
    as many aggregates as entries."""
    A = P.poisson2d(m)
    hub = m * (m // 2) + m // 2
    row = set(A.col[A.rowptr[hub]:A.rowptr[hub + 1]].tolist())
    far = [int(j) for j in np.random.default_rng(seed).permutation(A.n) if int(j) not in row][:degree]
    extra = {hub: [(j, -1e-3) for j in far]}
    extra.update({j: [(hub, -1e-3)] for j in far})
    rp, ci, va = [0], [], []
    for i in range(A.n):
        ent = list(zip(A.col[A.rowptr[i]:A.rowptr[i + 1]].tolist(), A.val[A.rowptr[i]:A.rowptr[i + 1]].tolist()))
        more = extra.get(i, [])
        ent = sorted([(j, v + (1e-3 * len(more) if j == i else 0.0)) for j, v in ent] + more)
        ci += [j for j, _ in ent]
        va += [v for _, v in ent]
        rp.append(len(ci))
    return P.CSR(A.n, np.array(rp, np.int32), np.array(ci, np.int32), np.array(va))


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("degree", [19, 20, 21, 40, 59, 60, 61, 124, 700])
def test_cycle_with_a_hub(env, prec, degree):
    """Rows of 24 to 705 entries: the hierarchy's arrays are consistent (the values of A P
    among them), and in FP64 the cycle is the oracle's."""
    amg, oracle = env
    A = hub_grid(48, degree, degree)
    b = P.rhs_uniform(A.n, 3)
    g = amg.Hierarchy(A, alpha=0.25, seed=1, precision=prec)
    assert amg.lib().amg_validate_hierarchy(g.h) == 0, amg.amg_last_error()
    z = g.precond(b)
    zo = oracle.Hierarchy(A, alpha=0.25, seed=1).precond(b)
    assert np.linalg.norm(z - zo) <= (1e-10, 1e-4, 1e-2)[prec] * np.linalg.norm(zo)
    x, info = g.solve(b, tol=1e-8)
    assert info["final_relres"] <= 1e-8
    amg.amg_resetup_values(g.h, 1.5 * A.val)
    assert amg.lib().amg_validate_hierarchy(g.h) == 0, amg.amg_last_error()


@pytest.mark.parametrize("prec", [0, 1])
def test_setup_time_of_a_long_row(env, prec):
    """A row of 3,000 entries costs a setup some walks along it by one thread (tens of
    dependent loads of under a microsecond each an entry: below 0.1 s), not one walk per
    entry (some 9 million steps, above 0.4 s)."""
    amg, _ = env
    A = hub_grid(160, 3000, 5)
    times = []
    for _ in range(3):
        g = amg.Hierarchy(A, alpha=0.25, seed=1, precision=prec)
        times.append(amg.amg_last_solve_info(g.h)["setup_ms"])
        g.free()
    print(f"precision {prec}: setup {min(times):.1f} ms")
    assert min(times) < 100.0
