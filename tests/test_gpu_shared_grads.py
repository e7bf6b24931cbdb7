"""One buffer as dX and dY of an accumulating backward: it receives both derivatives (a Gram
of X with itself, each argument's gradient wanted in the same place), in every form of the
backward.  FP32: both sides add the same terms to the same start in one of two orders, 1e-6 of
the largest; FP64 1e-14."""
import numpy as np
import pytest
import torch

from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu

# (paths, points, channels, dyadic order): band form with 2, 4 and 8 rows a lane, and pairs
# too long for it (strip form)
SHAPES = [(70, 40, 3, 0), (40, 90, 5, 1), (33, 200, 8, 1), (3, 700, 6, 1)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("variant", [sigk.Variant(), sigk.Variant(static_kernel="rbf")])
@pytest.mark.parametrize("gram", [True, False])
@pytest.mark.parametrize("B,L,d,lam", SHAPES)
def test_one_buffer_receives_both(B, L, d, lam, gram, variant, dtype):
    need_gpu()
    if L > 500 and (variant.static_kernel == "rbf" or dtype == torch.float64):
        pytest.skip("the plain backward; the shorter paths cover it")
    X = to_dev(inputs.random_paths(7100 + L, B, L, d, time_channel=True), dtype)
    Y = X if gram else to_dev(inputs.random_paths(7200 + L, B, L, d, time_channel=True), dtype)
    gen = np.random.default_rng(3)
    g = to_dev(gen.normal(size=(B, B) if gram else B), dtype)
    start = to_dev(gen.normal(size=X.shape), dtype)
    back = sigk.gram_backward if gram else sigk.pairs_backward
    dX, dY = back(g, X, Y, lam, variant=variant)
    want = start + dX + dY
    both = start.clone()
    back(g, X, Y, lam, variant=variant, dX=both, dY=both, accumulate=True)
    size = float((start.abs() + dX.abs() + dY.abs()).max())
    assert float((both - want).abs().max()) <= (1e-6 if dtype == torch.float32 else 1e-14) * size
