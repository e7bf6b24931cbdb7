"""The strip path's FP32 adjoint and its tiled chain rule (csrc/fwd_strip.cu,
csrc/tile_gemm.cuh): strips, 32-step chunks, groups of four windows and quads of
columns that begin and end everywhere, at every dyadic order, against the
oracle's gradient with the FP32 gradient tolerance (1e-4 of the largest entry)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


# (pairs, L, M, d, dyadic order, scheme)
@pytest.mark.parametrize("B,L,M,d,lam,scheme", [
    (2, 600, 2, 3, 0, "explicit"), (3, 37, 530, 5, 0, "explicit"), (1, 1100, 515, 33, 0, "implicit"),
    (2, 300, 259, 8, 1, "explicit"), (2, 34, 531, 2, 1, "explicit"), (1, 1030, 1025, 70, 1, "explicit"),
    (5, 261, 262, 32, 1, "implicit"), (2, 260, 131, 4, 2, "explicit"), (1, 400, 137, 64, 2, "implicit"),
    (2, 140, 70, 3, 3, "explicit"), (1, 131, 129, 6, 3, "implicit"), (70, 150, 3, 4, 1, "explicit"),
])
def test_strip_backward(B, L, M, d, lam, scheme):
    need_gpu()
    X32, X64 = inputs.f32(inputs.random_paths(9800 + L, B, L, d, time_channel=d > 2))
    Y32, Y64 = inputs.f32(inputs.random_paths(9900 + M, B, M, d, time_channel=d > 2))
    g32, g64 = inputs.f32(np.random.default_rng(3).normal(size=B))
    dX, dY = sigk.pairs_backward(to_dev(g32), to_dev(X32), to_dev(Y32), lam, rec=sigk.REC_STRIP,
                                 variant=sigk.Variant(scheme=scheme), check_status=True)
    rX, rY = oracle.pairs_grad(X64, Y64, lam, g64, scheme=scheme)
    for got, ref in ((dX, rX), (dY, rY)):
        assert torch.isfinite(got).all()
        assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-4 * np.max(np.abs(ref))
