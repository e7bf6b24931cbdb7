"""Calls of several host threads with different shapes: the shared memory that a kernel may
use is a setting of the kernel, so a thread with a small shape must not lower it between another
thread's setting and its launch (which then fails).  Threads repeat one shape each on streams
of their own, through the C entry points so that the calls do overlap; every call succeeds and
results are bit for bit those of a call alone."""
import ctypes
import threading

import pytest
import torch

from paper_2006_14794_gb300 import inputs, sigk

from .gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu

# (dtype, static kernel, order, two shapes of one kernel instance: little and much shared
# memory, calls a thread)
CASES = {"wave64, coefficients first": (torch.float64, 0, 1, [(4, 20, 24, 2), (4, 20, 150, 40)], 3000),
         "wave64, inline": (torch.float64, 0, 1, [(640, 100, 90, 2), (640, 100, 90, 60)], 300),
         "band coefficients": (torch.float32, 1, 2, [(20, 100, 110, 2), (20, 100, 128, 30)], 3000)}


@pytest.mark.parametrize("name", sorted(CASES))
def test_threads_with_other_shapes(name):
    need_gpu()
    dtype, kernel, lam, shapes, reps = CASES[name]
    lib, code = sigk.lib(), sigk.SIGK_F64 if dtype == torch.float64 else sigk.SIGK_F32
    o = sigk.SigkOpts()
    o.static_kernel, o.sigma = kernel, 1.0
    jobs = []
    for B, L, M, d in shapes * 2:
        X = to_dev(inputs.random_paths(6400 + L + d, B, L, d), dtype)
        Y = to_dev(inputs.random_paths(6500 + M + d, B, M, d), dtype)
        want = sigk.pairs(X, Y, lam, variant=sigk.Variant(static_kernel="rbf" if kernel else "linear"))
        n = lib.sigk_workspace_bytes(sigk.OP_PAIRS, B, 0, L, M, d, lam, code, ctypes.byref(o))
        ws = torch.empty(max(n, 1), dtype=torch.uint8, device="cuda")
        out = torch.zeros_like(want)
        stream = torch.cuda.Stream()
        args = (X.data_ptr(), Y.data_ptr(), B, L, M, d, lam, code, ctypes.byref(o), out.data_ptr(), ws.data_ptr(), n,
                stream.cuda_stream)
        jobs.append((args, X, Y, ws, out, want))
    torch.cuda.synchronize()
    status = [None] * len(jobs)
    gate = threading.Barrier(len(jobs))

    def work(i):
        call, args = lib.sigk_pairs, jobs[i][0]
        gate.wait()
        status[i] = {call(*args) for _ in range(reps)}

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert status == [{sigk.SIGK_OK}] * len(jobs)
    for _, _, _, _, out, want in jobs:
        assert torch.equal(out, want)
