"""Row features on rows the staged kernel treats specially: blocks with more
entries than its shared memory holds, explicit zeros, values at the ends of the
FP64 exponent range, more than eight and no off-diagonals.  Bit for bit the oracle's."""
import numpy as np
import pytest

from paper_1403_1649_gb300 import problems as P

pytestmark = pytest.mark.gpu


def matrix(n, widest, scale, seed):
    u = P.uniform01(seed, 0, 4 * n)
    rows = []
    for i in range(n):
        w = int(u[4 * i] * widest) if i % 5 else (0 if i % 2 else widest)
        cols = sorted({int((i + 1 + k * (1 + int(7 * u[4 * i + 1]))) % n) for k in range(w)} - {i})
        v = {c: (2.0 * P.uniform01(seed + 1 + i, 0, len(cols))[k] - 1.0) * scale for k, c in enumerate(cols)}
        for c in cols[::6]:
            v[c] = 0.0
        v[i] = scale * (1.0 + u[4 * i + 2]) * (-1.0 if i % 7 == 3 else 1.0)
        rows.append(sorted(v.items()))
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    return P.CSR(n, rp, np.array([c for r in rows for c, _ in r], np.int32), np.array([a for r in rows for _, a in r]))


@pytest.mark.parametrize("n,widest,scale", [(1, 0, 1.0), (127, 6, 1.0), (129, 15, 1.0), (300, 60, 1.0),
                                            (200, 9, 1e-290), (200, 9, 1e290), (200, 9, 2.0 ** -399)])
def test_features_bit_exact_on_special_rows(n, widest, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle
    from paper_1403_1649_gb300 import amg, build
    build.build()
    oracle.build()
    A = matrix(n, widest, scale, 21)
    # a one-level hierarchy: the row features do not depend on the rest of the setup
    h = amg.Hierarchy(A, alpha=0.25, seed=1, max_levels=1, symmetric=0, outer=1)
    f = np.zeros((n, 16), np.float32)
    assert amg.lib().amg_features(h.h, 0, f.ctypes.data, None) == 0
    assert np.array_equal(f, oracle.features(A, level=0))
