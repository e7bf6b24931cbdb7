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


def check_values_by_nodes(X, Y, lam, **kw):
    """Beside jumps k changes sign and size along the paths and may end near zero, where the
    oracle's own rounding reaches 1e-10 of it (against 80-bit arithmetic): 1e-11 of the largest
    node of the pair's solution, which is what the scheme's rounding is relative to."""
    kw = dict(RBF, **kw)
    got = sigk.pairs(dev(X), dev(Y), lam, variant=sigk.Variant(**kw)).cpu().numpy()
    k, nodes = oracle.pairs_surface(X, Y, lam, **kw)
    assert np.max(np.abs(got - k) / np.abs(nodes).max(axis=(1, 2))) <= 1e-11


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


def jumps(P, sizes, seed, stay):
    """Every path of P with one jump of each size (bandwidths) in a random direction at a random
    point: back at the next point, or for good."""
    rng = np.random.default_rng(seed)
    P = P.copy()
    for size in sizes:
        for b in range(P.shape[0]):
            at = rng.integers(1, P.shape[1])
            v = rng.normal(size=P.shape[2])
            P[b, at:None if stay else at + 1] += size * v / np.linalg.norm(v)
    return P


# jumps of X and of Y; None: Y is X, so that both jump together
JUMPS = [((6,), ()), ((9,), ()), ((3, 5), (5, 9)), ((20,), (6,)), ((60,), (45, 20)), ((6,), None), ((9, 5), None),
         ((20, 60), None)]


def jumping(B, L, M, d, sizes, stay):
    X = jumps(paths(9810 + L, B, L, d) + 0.5, sizes[0], 31, stay)
    if sizes[1] is None:
        return X, X
    return X, jumps(paths(9910 + M, B, M, d) + 0.5, sizes[1], 37, stay)


@pytest.mark.parametrize("stay", [False, True])
@pytest.mark.parametrize("sizes", JUMPS)
@pytest.mark.parametrize("B,L,M,d,lam", [FORWARD[0], FORWARD[2], FORWARD[3], FORWARD[4], FORWARD[5]])
def test_values_beside_jumps(B, L, M, d, lam, sizes, stay):
    need_gpu()
    check_values_by_nodes(*jumping(B, L, M, d, sizes, stay), lam)


@pytest.mark.parametrize("scheme", ["explicit", "implicit"])
@pytest.mark.parametrize("sizes", JUMPS)
@pytest.mark.parametrize("B,L,M,d,lam", BACKWARD[:3])
def test_gradients_beside_jumps(B, L, M, d, lam, sizes, scheme):
    need_gpu()
    check_gradients(*jumping(B, L, M, d, sizes, False), lam, scheme=scheme)


def test_equal_corners_off_a_far_one():
    """Cells whose other three corners are near one another: the exponents A and B are large and
    C cancels them; and cells whose two paths meet from far apart, where only C is large."""
    need_gpu()
    X, Y = paths(9821, 9, 30, 3), paths(9822, 9, 31, 3)
    for b in range(9):
        X[b, 10] += (5.0 + b, 0, 0)                  # x_10 far, x_11, y_q, y_{q+1} near
        Y[b, 20] += (-(5.0 + b) / 2, (5.0 + b) * 0.75 ** 0.5, 0)
        X[b, 21:] += ((5.0 + b) / 2, (5.0 + b) * 0.75 ** 0.5, 0)
    check_values_by_nodes(X, Y, 1)
    check_gradients(X[:3], Y[:3], 1)
