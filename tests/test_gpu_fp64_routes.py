"""What FP64 calls cost on the route they take by default, beside the general one-block-per-pair
kernels (REC_PLAIN): never much more, for shapes where the wavefront has little to gain.  Times
are the best of several on an idle stream; a factor of 1.25 allows for their spread."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, rel_err, to_dev

pytestmark = pytest.mark.gpu


def paths(seed, B, L, d):
    return to_dev(inputs.random_paths(seed, B, L, d, time_channel=d > 1), torch.float64)


def us(call, reps=5):
    call()
    best = 1e30
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        for _ in range(reps):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / reps)
    return best


def test_two_plain_blocks_share_a_multiprocessor():
    """The plain sweep is bound by its chain of diagonals: two pairs a multiprocessor take the
    time of one, if its registers let two blocks in."""
    need_gpu()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    X, Y = paths(71, 2 * sms, 24, 20), paths(72, 2 * sms, 160, 20)
    one = us(lambda: sigk.pairs(X[:sms], Y[:sms], 0, rec=sigk.REC_PLAIN))
    two = us(lambda: sigk.pairs(X, Y, 0, rec=sigk.REC_PLAIN))
    assert two <= 1.5 * one


# (pairs, L, M, d, dyadic order): one and two coarse rows, short sides, tiny grids
SHORT = [(1310, 5, 11, 9, 0), (1316, 2, 2, 2, 1), (628, 25, 11, 18, 0), (217, 83, 7, 17, 0), (1457, 4, 3, 32, 1)]


@pytest.mark.parametrize("kernel", ["linear", "rbf"])
@pytest.mark.parametrize("B,L,M,d,lam", SHORT)
def test_short_paths_backward(B, L, M, d, lam, kernel):
    need_gpu()
    X, Y = paths(73 + L, B, L, d), paths(74 + M, B, M, d)
    g = torch.ones(B, dtype=torch.float64, device="cuda")
    v = sigk.Variant(static_kernel=kernel)
    default = us(lambda: sigk.pairs_backward(g, X, Y, lam, variant=v))
    plain = us(lambda: sigk.pairs_backward(g, X, Y, lam, variant=v, rec=sigk.REC_PLAIN))
    assert default <= 1.25 * plain


# coarse rows around the steps that a sweep without virtual rows leaves out (8, 16, 24 lanes)
@pytest.mark.parametrize("kernel", ["linear", "rbf"])
@pytest.mark.parametrize("lam", [0, 1, 2, 3])
@pytest.mark.parametrize("nx", [1, 4, 7, 8, 9, 16, 24, 25, 31, 32, 33, 40, 70])
def test_virtual_rows_are_left_out(nx, lam, kernel):
    need_gpu()
    kw = dict(static_kernel=kernel, sigma=1.0)
    rng = np.random.default_rng(nx)
    for B, ny in ((3, nx), (5, nx + 30), (400, nx + 3)):
        if B > 5 and nx > 33:
            continue
        X = inputs.random_paths(75 + nx, B, nx + 1, 3, time_channel=True)
        Y = inputs.random_paths(76 + ny, B, ny + 1, 3, time_channel=True)
        Xd, Yd = to_dev(X, torch.float64), to_dev(Y, torch.float64)
        v = sigk.Variant(**kw)
        assert rel_err(sigk.pairs(Xd, Yd, lam, variant=v).cpu().numpy(), oracle.pairs(X, Y, lam, **kw)) <= 1e-11
        g = rng.normal(size=B)
        n = min(B, 8)   # the oracle's share
        got = sigk.pairs_backward(to_dev(g, torch.float64), Xd, Yd, lam, variant=v)
        for a, b in zip(got, oracle.pairs_grad(X[:n], Y[:n], lam, g[:n], **kw)):
            assert np.max(np.abs(a[:n].cpu().numpy() - b)) <= 1e-10 * np.max(np.abs(b))


# increments that leave a multiprocessor one block of one warp, with the lift at order 0
WIDE = [(195, 24, 161, 63, 0), (1200, 24, 161, 63, 0), (300, 60, 200, 50, 0), (150, 24, 161, 63, 0), (300, 20, 120, 90, 1)]


@pytest.mark.parametrize("kernel", ["linear", "rbf"])
@pytest.mark.parametrize("B,L,M,d,lam", WIDE)
def test_wide_paths_forward(B, L, M, d, lam, kernel):
    need_gpu()
    X, Y = paths(77 + L, B, L, d), paths(78 + M, B, M, d)
    v = sigk.Variant(static_kernel=kernel)
    default = us(lambda: sigk.pairs(X, Y, lam, variant=v), 1)
    plain = us(lambda: sigk.pairs(X, Y, lam, variant=v, rec=sigk.REC_PLAIN), 1)
    assert default <= 1.25 * plain
    n = 4
    want = oracle.pairs(X[:n].cpu().numpy(), Y[:n].cpu().numpy(), lam, static_kernel=kernel, sigma=1.0)
    assert rel_err(sigk.pairs(X, Y, lam, variant=v)[:n].cpu().numpy(), want) <= 1e-11


@pytest.mark.parametrize("rec", [sigk.REC_PLAIN, sigk.REC_CHAIN])
@pytest.mark.parametrize("size", [6.0, 9.0, 30.0])
def test_jumps_on_the_general_routes(size, rec):
    """A point of X and of Y some bandwidths off, apart and together: plain and strip sweeps."""
    need_gpu()
    kw = dict(static_kernel="rbf", sigma=1.0)
    X = inputs.random_paths(79, 6, 30, 3, time_channel=True) + 0.5
    Y = inputs.random_paths(80, 6, 33, 3, time_channel=True) + 0.5
    X[:3, 11] += size / 3 ** 0.5
    Y[:3, 20] -= size / 3 ** 0.5
    X[3:, 11:] += size / 3 ** 0.5
    Y[3:, 20:] += size / 3 ** 0.5
    got = sigk.pairs(to_dev(X, torch.float64), to_dev(Y, torch.float64), 1, rec=rec, variant=sigk.Variant(**kw))
    k, nodes = oracle.pairs_surface(X, Y, 1, **kw)
    assert np.max(np.abs(got.cpu().numpy() - k) / np.abs(nodes).max(axis=(1, 2))) <= 1e-11
