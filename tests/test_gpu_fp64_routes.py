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
