"""The FP32 RBF lift on data that is rough on the scale of the bandwidth, where the band
coefficients (csrc/band_coef.cu) cannot be carried from cell to cell: values for 2, 4 and 8
coarse rows a lane, channels staged at once and in chunks, both schemes; and what such a call
costs beside a smooth one.  Tolerance: FP32's 1e-5, of the largest node of the pair's solution
(k itself may end near zero, and the scheme's rounding is relative to its nodes)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu

# (rows a lane, dyadic order, L, M, d)
SHAPES = [(4, 1, 65, 66, 3), (4, 1, 40, 300, 33), (8, 1, 129, 130, 20), (8, 1, 70, 260, 65), (16, 1, 257, 258, 5),
          (16, 1, 150, 260, 130), (16, 2, 100, 128, 8), (16, 3, 65, 70, 35), (8, 0, 70, 75, 6), (4, 0, 60, 61, 40)]


def check(X, Y, R, lam, **kw):
    kw = dict(static_kernel="rbf", **kw)
    (X32, X64), (Y32, Y64) = inputs.f32(X), inputs.f32(Y)
    got = sigk.pairs(to_dev(X32), to_dev(Y32), lam, schedule=sigk.Schedule(rec=sigk.REC_BAND, rows_per_lane=R),
                     variant=sigk.Variant(**kw)).cpu().numpy()
    k, nodes = oracle.pairs_surface(X64, Y64, lam, **kw)
    assert np.max(np.abs(got - k) / np.abs(nodes).max(axis=(1, 2))) <= 1e-5


@pytest.mark.parametrize("scheme", ["explicit", "implicit"])
@pytest.mark.parametrize("sigma", [0.3, 0.1, 0.05])
@pytest.mark.parametrize("R,lam,L,M,d", SHAPES)
def test_small_bandwidths(R, lam, L, M, d, sigma, scheme):
    need_gpu()
    X = inputs.random_paths(4600 + L, 5, L, d, time_channel=True) + 0.5
    Y = inputs.random_paths(4700 + M, 5, M, d, time_channel=True) + 0.5
    check(X, Y, R, lam, sigma=sigma, scheme=scheme)


@pytest.mark.parametrize("R,lam,L,M,d", SHAPES[:7:2])
def test_paths_that_meet_from_far_apart(R, lam, L, M, d):
    """Three corners of a cell at equal distances: A and B near zero, C hundreds of bandwidths."""
    need_gpu()
    X = inputs.random_paths(4800 + L, 5, L, d, time_channel=True)
    Y = inputs.random_paths(4900 + M, 5, M, d, time_channel=True)
    for b, far in enumerate((3.0, 6.0, 12.0, 18.0, 25.0)):
        Y[b, :20, 0] += far
        X[b, 30:, 0] += far / 2
        X[b, 30:, 1] += far * 0.75 ** 0.5
        Y[b, 20:, 0] += far / 2
        Y[b, 20:, 1] += far * 0.75 ** 0.5
    check(X, Y, R, lam, sigma=1.0)


@pytest.mark.parametrize("B,L,d,lam", [(128, 128, 8, 2), (64, 128, 64, 0)])
def test_rough_data_costs_a_small_factor(B, L, d, lam):
    """The same Gram with bandwidths of 1 and of 0.2: four exponentials and series a cell against
    one series, about twice the call; cells formed with loads of their own take 7 to 35 times."""
    need_gpu()
    X = to_dev(inputs.random_paths(4950, B, L, d, time_channel=True))
    Y = to_dev(inputs.random_paths(4951, B, L, d, time_channel=True))

    def ms(sigma):
        v = sigk.Variant(static_kernel="rbf", sigma=sigma)
        times = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            sigk.gram(X, Y, lam, variant=v)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert ms(0.2) <= 5 * ms(1.0)


@pytest.mark.parametrize("R,lam,L,M,d", SHAPES[1:8:2])
@pytest.mark.parametrize("far", [50.0, 3000.0, 1e5])
def test_single_points_out_of_reach(R, lam, L, M, d, far):
    """Spikes of X away from Y and back: the exponents beside them cancel to nothing (and from
    1e7 on are no longer exact to one), while their neighbours' count."""
    need_gpu()
    X = inputs.random_paths(5000 + L, 5, L, d, time_channel=True)
    Y = inputs.random_paths(5100 + M, 5, M, d, time_channel=True)
    for b in range(5):
        X[b, 5 + 3 * b, 0] += far
        Y[b, 11 + 2 * b, 1] -= far
    check(X, Y, R, lam, sigma=1.0)
    check(X, Y, R, lam, sigma=0.2)
