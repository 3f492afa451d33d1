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


def exact_layer1(rows, w3, feat, dout):
    """Network with W1 = 0, W2 = 1, zero biases and powers of two w3 in the first output:
    the hidden activations are zero, dz1 = dz2 = w3 x dout exactly, and the gradients of
    W1, b1 and b2 are sums of products of the given FP32 values."""
    from oracle import oracle
    w = np.zeros(oracle.NPARAM, np.float32)
    w[1088:5184] = np.eye(64, dtype=np.float32).ravel()
    w[5248:5312] = w3
    dz = [[float(w3[u]) * float(dout[r, 0]) for u in range(64)] for r in range(rows)]
    return w, dz


@pytest.mark.parametrize("rows", [64, 150])
@pytest.mark.parametrize("mix", ["large_in_one_row", "tiny_unit", "tiny_rows", "zero_feature"])
def test_weight_gradients_of_mixed_magnitudes(rows, mix):
    """Tiles in which some products lie far outside the range of FP32 and others do not:
    every parameter's sum is that of its own terms, to 1e-13 of their magnitudes."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle
    from paper_1403_1649_gb300 import amg, build
    build.build()
    oracle.build()
    rng = np.random.default_rng(rows)
    feat = rng.uniform(0.1, 1.0, (rows, 16)).astype(np.float32)
    dout = rng.normal(size=(rows, 3)).astype(np.float32)
    w3 = np.zeros(64, np.float32)
    w3[0], w3[9] = 1.0, 0.5
    if mix == "large_in_one_row":
        feat[5, 3], dout[5, 0] = 1e25, 1e20
    elif mix == "tiny_unit":  # products of about 1e-42 beside ordinary ones
        w3[9] = 2.0 ** -70
        feat[:, 2] *= np.float32(1e-21)
    elif mix == "tiny_rows":  # one ordinary row among rows whose factors are tiny
        feat[1:, 4] *= np.float32(1e-22)
        feat[0, 4] = 0.0
        dout[1:, 0] *= np.float32(1e-22)
    else:
        feat[:, 7] = 0.0
        feat[1:, 8] = 0.0
    w, dz = exact_layer1(rows, w3, feat, dout)
    dev = torch.device("cuda")
    wd, fd, dd = (torch.from_numpy(a).to(dev) for a in (w, feat, dout))
    grad = torch.full((oracle.NPARAM,), np.nan, dtype=torch.float64, device=dev)
    assert amg.lib().amg_mlp_backward(rows, C.c_void_p(wd.data_ptr()), C.c_void_p(fd.data_ptr()),
                                      C.c_void_p(dd.data_ptr()), C.c_void_p(grad.data_ptr()), None) == 0
    torch.cuda.synchronize()
    g = grad.cpu().numpy()
    assert np.isfinite(g).all()
    for u in range(64):
        col = [dz[r][u] for r in range(rows)]
        for got in (g[1024 + u], g[5184 + u]):  # b1, b2
            assert abs(got - math.fsum(col)) <= 1e-13 * math.fsum(map(abs, col)), (u, got)
        for k in range(16):
            # products of two FP32 values are exact in FP64
            terms = [col[r] * float(feat[r, k]) for r in range(rows)]
            got = g[16 * u + k]
            assert abs(got - math.fsum(terms)) <= 1e-13 * math.fsum(map(abs, terms)), (u, k, got, math.fsum(terms))
