"""Kernels of the cycle at the sizes where they can go wrong: products on small
levels whose rows are shared by several warps (rows of 0 to ~150 entries, ragged
last slices), and cycles over aggregates of several dozen rows."""
import numpy as np
import pytest

from paper_1403_1649_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_1649_gb300 import amg, build
    build.build()
    amg.lib()
    return amg


@pytest.fixture(scope="session")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


def symmetric(n, pairs, seed):
    """Diagonally dominant symmetric matrix with the given off-diagonal positions."""
    pairs = sorted({(min(i, j), max(i, j)) for i, j in pairs if i != j})
    v = -(0.5 + P.uniform01(seed, 2, len(pairs)))
    rows = [[] for _ in range(n)]
    for (i, j), a in zip(pairs, v):
        rows[i].append((j, a))
        rows[j].append((i, a))
    rp, ci, va = [0], [], []
    for i in range(n):
        ent = sorted(rows[i] + [(i, 0.25 + sum(abs(a) for _, a in rows[i]))])
        ci += [j for j, _ in ent]
        va += [a for _, a in ent]
        rp.append(len(ci))
    return P.CSR(n, np.array(rp, np.int32), np.array(ci, np.int32), np.array(va, np.float64))


def wide_rows(n, widest, seed):
    """Rows of very different length: every 40th row reaches `widest` others."""
    u = P.uniform01(seed, 0, n * 3)
    pairs = [(i, int(u[3 * i + k] * n)) for i in range(0, n, 2) for k in range(3)]
    for i in range(0, n, 40):
        pairs += [(i, (i + 1 + 7 * k) % n) for k in range(min(widest, n - 1))]
    return symmetric(n, pairs, seed)


def stars(hubs, leaves, seed):
    """Hubs in a ring, each with its own leaves: aggregates of about `leaves` rows."""
    n = hubs * (leaves + 1)
    pairs = [(q * (leaves + 1), ((q + 1) % hubs) * (leaves + 1)) for q in range(hubs)]
    pairs += [(q * (leaves + 1), q * (leaves + 1) + 1 + k) for q in range(hubs) for k in range(leaves)]
    return symmetric(n, pairs, seed)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n,widest", [(33, 20), (257, 40), (1000, 150), (4001, 9)])
def test_spmv_wide_rows(gpu, prec, n, widest):
    """Every level's product element by element: FP64 within the rounding of its
    accumulation, FP32 and BF16 within that of the stored values too ((w + 4) u32
    sum |a x| for the FP32 sums of a row of w entries, u sum |a| (|x_j| + |x_i|)
    for values rounded to u and moved onto the diagonal)."""
    import torch
    A = wide_rows(n, widest, 5)
    g = gpu.Hierarchy(A, alpha=0.25, seed=3, precision=prec, coarse_max=8)
    for k in range(g.nlevels):
        L = g.level(k)
        Ak = P.CSR(L["n"], L["rowptr"], L["col"], L["val"])
        x = P.rhs_uniform(Ak.n, 50 + k).astype(np.float64 if prec == 0 else np.float32)
        xd = torch.from_numpy(x).cuda()
        yd = torch.full_like(xd, 7.0)
        gpu.amg_spmv(g.h, k, xd, yd)
        torch.cuda.synchronize()
        x64 = x.astype(np.float64)
        rows = np.repeat(np.arange(Ak.n), np.diff(Ak.rowptr))
        w = np.diff(Ak.rowptr) + 4.0
        term = np.bincount(rows, weights=np.abs(Ak.val * x64[Ak.col]), minlength=Ak.n)
        bound = w * 2.0 ** (-53 if prec == 0 else -24) * term + 1e-300
        if prec:
            off = Ak.col != rows
            moved = (np.abs(Ak.val) * (np.abs(x64[Ak.col]) + np.abs(x64[rows])))[off]
            bound += 2.0 ** (-24 if prec == 1 else -8) * np.bincount(rows[off], weights=moved, minlength=Ak.n)
        err = np.abs(yd.cpu().numpy().astype(np.float64) - Ak.matvec(x64))
        assert (err <= 2 * bound).all(), (k, (err / bound).max())


@pytest.mark.parametrize("hubs,leaves", [(40, 15), (60, 16), (30, 17), (24, 70)])
def test_cycle_over_large_aggregates(gpu, orc, hubs, leaves):
    """Aggregates around and beyond the members a lane group loads ahead (16): the
    FP64 cycle agrees with the oracle's to 1e-11, with and without a second level
    below, and reduced precisions reach the tolerance."""
    A = stars(hubs, leaves, 9)
    b = P.rhs_uniform(A.n, 19)
    for cmax in (8, 2 * hubs):
        g = gpu.Hierarchy(A, alpha=0.25, seed=2, coarse_max=cmax)
        o = orc.Hierarchy(A, alpha=0.25, seed=2, coarse_max=cmax)
        assert g.nlevels == o.nlevels
        assert np.bincount(g.level(0)["agg"]).max() > min(leaves, 16)
        zg, zo = g.precond(b), o.precond(b)
        assert np.linalg.norm(zg - zo) <= 1e-11 * np.linalg.norm(zo)
    for prec in (1, 2):
        _, info = gpu.Hierarchy(A, alpha=0.25, seed=2, coarse_max=8, precision=prec).solve(b, tol=1e-8)
        assert info["final_relres"] <= 1e-8


@pytest.mark.parametrize("t", [0.0, 5e-5, 2e-4, 0.25, 50.0])
@pytest.mark.parametrize("outer", [0, 1])
@pytest.mark.parametrize("m", [6, 61])
def test_inner_step_threshold(gpu, orc, t, outer, m):
    """The test of Alg. 5 from the product's sums and, for thresholds below 1e-4, from
    r~ itself: always, never and by the data, in the CG and GMRES variants, on levels
    of one and of several blocks; the cycle to 1e-10 of the oracle's."""
    A = P.varcoef2d(m, 4)
    b = P.rhs_uniform(A.n, 29)
    kw = dict(alpha=0.25, seed=2, coarse_max=4, kcycle_t=t, outer=outer)
    zg, zo = gpu.Hierarchy(A, **kw).precond(b), orc.Hierarchy(A, **kw).precond(b)
    assert np.linalg.norm(zg - zo) <= 1e-10 * np.linalg.norm(zo)


def test_second_step_test_with_sums_that_overflow(gpu, orc):
    """Matrix and right-hand side scaled by powers of two until r.r overflows in FP64
    while the step length stays finite: the test of Alg. 5 compares infinities and takes
    the first step, as the oracle does."""
    A = P.varcoef2d(60, 3)
    big = P.CSR(A.n, A.rowptr, A.col, np.ldexp(A.val, 600))
    b = np.ldexp(P.rhs_uniform(A.n, 4), 530)
    z = gpu.Hierarchy(big, alpha=0.25, seed=1).precond(b)
    zo = orc.Hierarchy(big, alpha=0.25, seed=1).precond(b)
    assert np.isfinite(zo).all() and np.isfinite(z).all()
    s = np.ldexp(1.0, 70)
    assert np.linalg.norm(s * z - s * zo) <= 1e-10 * np.linalg.norm(s * zo)


@pytest.mark.parametrize("prec,wave", [(0, 456), (1, 608), (2, 608)])
def test_reported_blocks_are_those_of_the_launches(gpu, prec, wave):
    """Levels of 3,082 and 6,329 slices: the launches with inner products run one wave of their
    kernel (three or four blocks on each of 152 SMs), tuned or not at most that."""
    A = P.poisson2d(314)
    n0 = gpu.Hierarchy(A, alpha=0.25, precision=prec).info()[0]
    assert (n0["n"] + 31) // 32 > 2048 and n0["spmv_blocks"] == min(wave, ((n0["n"] + 31) // 32 + 7) // 8)
    big = P.poisson2d(450)
    assert gpu.Hierarchy(big, alpha=0.25, precision=prec).info()[0]["spmv_blocks"] == wave
    assert gpu.Hierarchy(big, alpha=0.25, precision=prec, autotune=1).info()[0]["spmv_blocks"] <= wave
