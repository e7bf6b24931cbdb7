"""The column role's chain-rule contraction (band_cols_kernel, csrc/band.cu) where
its tiling can go wrong: 4 and 8 coarse rows a lane, rows that fill the band and
rows that leave part of a lane virtual, one and several 128-column tiles with and
without a remainder, channel counts around its blocks of 32; Grams with both
gradients (split reductions), symmetric Grams and pairs.
Tolerance: the FP32 gradient one of the other tests (1e-4 of the largest entry)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu

# (rows a lane, dyadic order, L, M, d): L - 1 of 32 R / 2^order coarse rows are real
SHAPES = [(8, 1, 129, 130, 33), (8, 1, 70, 300, 1), (4, 0, 100, 129, 5), (16, 2, 100, 128, 31),
          (16, 1, 257, 258, 32), (16, 1, 150, 160, 7), (8, 0, 200, 300, 65)]


def close(got, ref):
    got = got.double().cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))


@pytest.mark.parametrize("R,lam,L,M,d", SHAPES)
def test_column_gradients(R, lam, L, M, d):
    need_gpu()
    sched = sigk.Schedule(rec=sigk.REC_BAND, rows_per_lane=R)
    X32, X64 = inputs.f32(inputs.random_paths(5100 + L, 3, L, d, time_channel=d > 1))
    Y32, Y64 = inputs.f32(inputs.random_paths(5200 + M, 4, M, d, time_channel=d > 1))
    rng = np.random.default_rng(5)
    g = rng.normal(size=(3, 4))
    rX, rY = oracle.gram_grad(X64, Y64, lam, g)
    dX, dY = sigk.gram_backward(to_dev(g, torch.float32), to_dev(X32), to_dev(Y32), lam, schedule=sched)
    close(dX, rX)
    close(dY, rY)
    gp = rng.normal(size=3)
    rX, rY = oracle.pairs_grad(X64, Y64[:3], lam, gp)
    dX, dY = sigk.pairs_backward(to_dev(gp, torch.float32), to_dev(X32), to_dev(Y32[:3]), lam, schedule=sched)
    close(dX, rX)
    close(dY, rY)
    gs = rng.normal(size=(3, 3))
    rA, rB = oracle.gram_grad(X64, X64, lam, gs)
    dS, _ = sigk.gram_backward(to_dev(gs, torch.float32), to_dev(X32), to_dev(X32), lam, schedule=sched,
                               symmetric=True)
    close(dS, rA + rB)
