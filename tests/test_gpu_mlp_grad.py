"""Weight gradients of the smoother network at the tile edges of its kernel (64 rows
a tile, a block's second tile from 304 tiles on) and with back-propagated signals so
large or small that their FP32 products leave the range in which the paired sums are
exact enough (those tiles are summed in FP64)."""
import ctypes as C
import math

import numpy as np
import pytest

from paper_1403_1649_gb300 import problems as P
from test_gpu_learned import gradient_term_magnitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,scale", [(1, 1.0), (63, 1.0), (64, 1.0), (65, 1.0), (1000, 1.0), (304 * 64 + 5, 1.0),
                                        (130, 1e32), (130, 1e-32)])
def test_weight_gradients_at_tile_edges(rows, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle
    from paper_1403_1649_gb300 import amg, build
    build.build()
    oracle.build()
    rng = np.random.default_rng(rows)
    w = (rng.normal(size=oracle.NPARAM) * 0.2).astype(np.float32)
    feat = np.resize(oracle.features(P.fem2d(30, 4)), (rows, 16)).astype(np.float32)
    dout = (rng.normal(size=(rows, 3)) * scale).astype(np.float32)
    dev = torch.device("cuda")
    wd, fd, dd = (torch.from_numpy(a).to(dev) for a in (w, feat, dout))
    grad = torch.full((oracle.NPARAM,), np.nan, dtype=torch.float64, device=dev)
    assert amg.lib().amg_mlp_backward(rows, C.c_void_p(wd.data_ptr()), C.c_void_p(fd.data_ptr()),
                                      C.c_void_p(dd.data_ptr()), C.c_void_p(grad.data_ptr()), None) == 0
    torch.cuda.synchronize()
    g = grad.cpu().numpy()
    gref, _ = oracle.mlp_backward(w.astype(np.float64), feat, dout.astype(np.float64))
    S = gradient_term_magnitudes(w.astype(np.float64), feat.astype(np.float64), dout.astype(np.float64))
    assert (np.abs(g - gref) <= 2e-5 * S).all(), (np.abs(g - gref) / (S + 1e-300)).max()
    # the output biases' gradients are sums of the given FP32 values: FP64 results
    for q in range(3):
        col = [float(v) for v in dout[:, q]]
        assert abs(g[oracle.NPARAM - 3 + q] - math.fsum(col)) <= 1e-13 * math.fsum(map(abs, col))
