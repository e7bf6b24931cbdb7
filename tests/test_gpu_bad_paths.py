"""A path with a NaN or an infinity at one of its ends spoils its own pairs only: the band
form's chains of pairs pass through padding columns between one pair and the next, whose
coefficients are zero whatever the points.  The other pairs' values and gradients are bit for
bit those of the batch without the bad path."""
import numpy as np
import pytest
import torch

from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu

# (pairs, L, M, d, dyadic order): 2, 4 and 8 coarse rows a lane, columns that do not fill the
# last macro-step, more pairs than the card has warps (chains of several)
SHAPES = [(6000, 12, 14, 3, 1), (6000, 20, 40, 5, 0), (3000, 70, 75, 4, 1), (3000, 180, 190, 3, 1), (2500, 40, 42, 40, 1)]


@pytest.mark.parametrize("kernel", ["linear", "rbf"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("B,L,M,d,lam", SHAPES)
def test_bad_paths_spoil_their_own_pairs_only(B, L, M, d, lam, bad, kernel):
    need_gpu()
    X = inputs.random_paths(6100 + L, B, L, d, time_channel=True)
    Y = inputs.random_paths(6200 + M, B, M, d, time_channel=True)
    variant = sigk.Variant(static_kernel=kernel)
    g = to_dev(np.random.default_rng(5).normal(size=B))
    rows = np.random.default_rng(6).choice(B, size=40, replace=False)
    good = np.ones(B, bool)
    good[rows] = False
    Xb, Yb = X.copy(), Y.copy()
    Yb[rows[:10], 0, 0] = bad
    Yb[rows[10:20], -1, 1] = bad
    Xb[rows[20:30], 0, 0] = bad
    Xb[rows[30:], -1, 1] = bad
    keep = torch.as_tensor(good).cuda()
    for a, b in ((X, Xb), (X, X)):   # the bad paths among the longer side's or the shorter side's
        ca, cb = to_dev(a), to_dev(Y)
        ba, bb = to_dev(b), to_dev(Yb)
        k, kb = sigk.pairs(ca, cb, lam, variant=variant), sigk.pairs(ba, bb, lam, variant=variant)
        assert torch.equal(k[keep], kb[keep])
        for u, v in zip(sigk.pairs_backward(g, ca, cb, lam, variant=variant),
                        sigk.pairs_backward(g, ba, bb, lam, variant=variant)):
            assert torch.isfinite(v[keep]).all()
            if kernel == "linear":
                assert torch.equal(u[keep], v[keep])


@pytest.mark.parametrize("kernel", ["linear", "rbf"])
def test_the_surface_keeps_its_border(kernel):
    """Row and column 0 are 1 whatever the path."""
    need_gpu()
    X = inputs.random_paths(6301, 40, 30, 3, time_channel=True)
    Y = inputs.random_paths(6302, 40, 38, 3, time_channel=True)
    Y[7, 0, 1] = float("nan")
    _, surf = sigk.pairs_surface(to_dev(X), to_dev(Y), 1, rec=sigk.REC_BAND, variant=sigk.Variant(static_kernel=kernel))
    assert torch.equal(surf[:, 0], torch.ones_like(surf[:, 0]))
    assert torch.equal(surf[:, :, 0], torch.ones_like(surf[:, :, 0]))
