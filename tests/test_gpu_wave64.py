"""FP64 pairs of uniform lengths on the register wavefront (csrc/wave64.cu):
every (coarse rows a lane, dyadic order) family around the edges of its bands,
one warp and several, blocks of a cluster, both orientations, both schemes and
the RBF lift, against the oracle.  The tolerances are the FP64 ones of the
other tests (1e-11 for values, 1e-10 for gradients)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, rel_err, to_dev

pytestmark = pytest.mark.gpu

VARIANTS = {"explicit": {}, "implicit": dict(scheme="implicit"), "rbf": dict(static_kernel="rbf", sigma=0.8)}


def paths(seed, B, L, d):
    return inputs.random_paths(seed, B, L, d, scale=1.5, time_channel=d > 1)


def dev(a):
    return to_dev(a, torch.float64)


# (pairs, L, M, d, dyadic order): 32 NG coarse rows a warp, +-1; one column;
# few pairs of many rows (several warps and cluster blocks), many pairs
SHAPES = [(3, 2, 2, 1, 0), (5, 33, 40, 3, 0), (4, 34, 34, 2, 0), (2, 2, 90, 4, 1), (7, 32, 33, 5, 1),
          (3, 66, 64, 3, 1), (2, 97, 150, 2, 1), (1, 300, 513, 3, 0), (2, 260, 200, 7, 1), (1, 129, 130, 8, 2),
          (2, 128, 97, 4, 2), (3, 65, 20, 3, 2), (1, 40, 41, 2, 3), (2, 70, 65, 3, 3), (700, 20, 18, 3, 1),
          (650, 130, 128, 2, 0)]


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("B,L,M,d,lam", SHAPES)
def test_forward(B, L, M, d, lam, variant):
    need_gpu()
    X, Y = paths(9100 + L, B, L, d), paths(9200 + M, B, M, d)
    got = sigk.pairs(dev(X), dev(Y), lam, variant=sigk.Variant(**VARIANTS[variant])).cpu().numpy()
    assert rel_err(got, oracle.pairs(X, Y, lam, **VARIANTS[variant])) <= 1e-11


@pytest.mark.parametrize("symmetric", [False, True])
def test_gram(symmetric):
    need_gpu()
    X, Y = paths(9301, 9, 50, 4), paths(9302, 14, 37, 4)
    if symmetric:
        Y = X
    got = sigk.gram(dev(X), dev(Y), 2, symmetric=symmetric).cpu().numpy()
    assert rel_err(got, oracle.gram(X, Y, 2)) <= 1e-11


def close(got, ref):
    got = got.cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("B,L,M,d,lam", [s for s in SHAPES if s[0] <= 7] + [(400, 20, 18, 3, 1)])
def test_backward(B, L, M, d, lam, variant):
    need_gpu()
    kw = VARIANTS[variant]
    X, Y = paths(9400 + L, B, L, d), paths(9500 + M, B, M, d)
    g = np.random.default_rng(7).normal(size=B)
    dX, dY = sigk.pairs_backward(dev(g), dev(X), dev(Y), lam, variant=sigk.Variant(**kw))
    rX, rY = oracle.pairs_grad(X, Y, lam, g, **kw)
    close(dX, rX)
    close(dY, rY)


def test_gram_backward_one_side_accumulates():
    need_gpu()
    X, Y = paths(9601, 5, 45, 6), paths(9602, 7, 30, 6)
    g = np.random.default_rng(8).normal(size=(5, 7))
    rX, rY = oracle.gram_grad(X, Y, 1, g)
    start = np.random.default_rng(9).normal(size=X.shape)
    dX, none = sigk.gram_backward(dev(g), dev(X), dev(Y), 1, need_dy=False, dX=dev(start), accumulate=True)
    assert none is None
    close(dX, start + rX)
    _, dY = sigk.gram_backward(dev(g), dev(X), dev(Y), 1, need_dx=False)
    close(dY, rY)


def test_backward_in_a_small_workspace():
    """One slot only (the grid shrinks to it), then none: the call is refused as before."""
    need_gpu()
    import ctypes
    B, L, d, lam = 6, 24, 3, 1
    X, Y = paths(9701, B, L, d), paths(9702, B, L, d)
    g = np.random.default_rng(10).normal(size=B)
    rX, rY = oracle.pairs_grad(X, Y, lam, g)
    o, lib = sigk.SigkOpts(), sigk.lib()
    need = lib.sigk_workspace_bytes(sigk.OP_PAIRS_BACKWARD, B, 0, L, L, d, lam, 1, ctypes.byref(o))
    Xd, Yd, gd = dev(X), dev(Y), dev(g)
    dX, dY = torch.empty_like(Xd), torch.empty_like(Yd)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    for size, want in ((need, 0), (need // B, 0), (0, sigk.SIGK_ENOMEM_WS)):
        st = lib.sigk_pairs_backward(gd.data_ptr(), Xd.data_ptr(), Yd.data_ptr(), B, L, L, d, lam, 1,
                                     ctypes.byref(o), dX.data_ptr(), dY.data_ptr(), ws.data_ptr(), size,
                                     torch.cuda.current_stream().cuda_stream)
        assert st == want
        if want == 0:
            close(dX, rX)
            close(dY, rY)
