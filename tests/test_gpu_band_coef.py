"""The band coefficients (csrc/band_coef.cu) where their tiling can go wrong:
2, 4 and 8 coarse rows a lane, one and several units a pair, more channels than
are staged at once, rows that exactly fill the band, and for the RBF lift paths
with jumps of many bandwidths (slots formed cell by cell beside carried ones).
Tolerance: the FP32 one of the other tests (1e-5 relative to max(|k|, 1e-3))."""
import numpy as np
import pytest

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, rel_err, to_dev

pytestmark = pytest.mark.gpu

# (rows a lane, dyadic order, L, M, d)
SHAPES = [(4, 1, 65, 66, 3), (4, 1, 40, 300, 33), (8, 1, 129, 130, 20), (8, 1, 70, 500, 65), (16, 1, 257, 258, 5),
          (16, 1, 200, 700, 40), (16, 1, 150, 260, 130), (16, 2, 100, 128, 8), (16, 3, 65, 70, 35)]


def close(X, Y, R, lam, variant):
    (X32, X64), (Y32, Y64) = inputs.f32(X), inputs.f32(Y)
    got = sigk.gram(to_dev(X32), to_dev(Y32), lam, schedule=sigk.Schedule(rec=sigk.REC_BAND, rows_per_lane=R),
                    variant=sigk.Variant(**variant)).cpu().numpy()
    assert rel_err(got, oracle.gram(X64, Y64, lam, **variant)) <= 1e-5


@pytest.mark.parametrize("variant", [{}, dict(static_kernel="rbf", sigma=1.0),
                                     dict(static_kernel="rbf", sigma=0.7, scheme="implicit")])
@pytest.mark.parametrize("R,lam,L,M,d", SHAPES)
def test_band_coefficients(R, lam, L, M, d, variant):
    need_gpu()
    X = inputs.random_paths(4100 + L, 3, L, d, time_channel=True)
    Y = inputs.random_paths(4200 + M, 4, M, d, time_channel=True)
    close(X, Y, R, lam, variant)


@pytest.mark.parametrize("R,lam,L,M,d", SHAPES[:6:2])
def test_lift_with_jumps(R, lam, L, M, d):
    """Points 0.5 to 1.5 bandwidths off and back, which leave the kernels of order one: slots
    with exponents above the carried form's limit beside slots below it.  About 800 cells lie
    beside a jump; FP32 coefficients of at most 0.9 there, off by 2e-7 each and at random, move
    k by about 2e-6."""
    need_gpu()
    X = inputs.random_paths(4300 + L, 3, L, d, time_channel=True)
    Y = inputs.random_paths(4400 + M, 4, M, d, time_channel=True)
    rng = np.random.default_rng(11)
    for P in (X, Y):
        for size in (0.5, 1.0, 1.5):
            for b in range(P.shape[0]):
                P[b, rng.integers(1, P.shape[1])] += size / np.sqrt(d)
    close(X, Y, R, lam, dict(static_kernel="rbf", sigma=1.0))


def test_lift_with_far_jumps_is_finite():
    """Jumps of 20 bandwidths: kappa underflows on one side of a cell and its ratio overflows;
    the product of the two must not become a NaN."""
    need_gpu()
    X = inputs.random_paths(4501, 3, 60, 3, time_channel=True)
    Y = inputs.random_paths(4502, 4, 70, 3, time_channel=True)
    X[:, 20] += 20.0
    Y[:, 33] += 15.0
    k = sigk.gram(to_dev(X), to_dev(Y), 1, variant=sigk.Variant(static_kernel="rbf", sigma=1.0)).cpu().numpy()
    assert np.isfinite(k).all()
