"""The RBF lift in FP64 (csrc/wave64.cu) on paths as users have them: first points
anywhere, jumps of many bandwidths.  Values and gradients against the oracle, at the FP64
tolerances of the other tests (1e-11 and 1e-10); the lift sees differences of points only, so
neither depends on where the paths lie."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, rel_err, to_dev

pytestmark = pytest.mark.gpu

RBF = dict(static_kernel="rbf", sigma=1.0)
# (pairs, L, M, d, dyadic order): coefficients formed first (few pairs: one coarse row a
# lane) and in the sweep with 2 and 4 rows a lane; even lengths leave an odd number of
# virtual rows, so a lane holds virtual and real ones; odd ones with none
FORWARD = [(8, 100, 97, 3, 1), (3, 40, 41, 2, 3), (600, 50, 53, 3, 1), (580, 100, 98, 3, 0), (580, 100, 98, 3, 1),
           (580, 128, 100, 2, 2), (580, 65, 66, 3, 2), (580, 50, 48, 2, 3)]
BACKWARD = [(5, 40, 37, 3, 1), (3, 33, 50, 2, 0), (4, 34, 20, 5, 2), (2, 20, 21, 3, 3)]


def paths(seed, B, L, d):
    return inputs.random_paths(seed, B, L, d, scale=1.5, time_channel=True)


def dev(a):
    return to_dev(a, torch.float64)


def check_values(X, Y, lam, **kw):
    kw = dict(RBF, **kw)
    got = sigk.pairs(dev(X), dev(Y), lam, variant=sigk.Variant(**kw)).cpu().numpy()
    assert rel_err(got, oracle.pairs(X, Y, lam, **kw)) <= 1e-11


def check_gradients(X, Y, lam, **kw):
    kw = dict(RBF, **kw)
    g = np.random.default_rng(17).normal(size=X.shape[0])
    got = sigk.pairs_backward(dev(g), dev(X), dev(Y), lam, variant=sigk.Variant(**kw))
    for a, b in zip(got, oracle.pairs_grad(X, Y, lam, g, **kw)):
        assert np.max(np.abs(a.cpu().numpy() - b)) <= 1e-10 * np.max(np.abs(b))


# what is added to every point of X and of Y
OFFSETS = [(0.5, 0.5), (-5.0, -4.6), (1000.0, 1000.3), (20000.0, 20000.0)]


@pytest.mark.parametrize("shift", OFFSETS)
@pytest.mark.parametrize("B,L,M,d,lam", FORWARD)
def test_values_wherever_the_paths_start(B, L, M, d, lam, shift):
    need_gpu()
    check_values(paths(9800 + L, B, L, d) + shift[0], paths(9900 + M, B, M, d) + shift[1], lam)


@pytest.mark.parametrize("shift", OFFSETS)
@pytest.mark.parametrize("B,L,M,d,lam", BACKWARD)
def test_gradients_wherever_the_paths_start(B, L, M, d, lam, shift):
    need_gpu()
    check_gradients(paths(9850 + L, B, L, d) + shift[0], paths(9950 + M, B, M, d) + shift[1], lam)
