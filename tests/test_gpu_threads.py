"""Calls from several host threads at once.  Calls of one device take turns on its
workspace, but a plan has its own and the no-allocation call has the caller's
buffers, so their launches come between a larger call's: the shared memory that
one launch asks for must not be taken away by another."""
import ctypes as C
import math
import threading

import numpy as np
import pytest

from paper_1908_02518_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROUNDS = 300


def _together(*loops):
    """Runs the loops on a thread each until the first one ends; their errors."""
    errors, done = [], threading.Event()

    def run(loop, lead):
        try:
            loop(done)
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(repr(e))
        finally:
            if lead:
                done.set()

    threads = [threading.Thread(target=run, args=(f, q == 0)) for q, f in enumerate(loops)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def _calls(n):
    import torch
    import paper_1908_02518_gb300 as rg
    x = torch.from_numpy(W.distance_matrix(W.cube_points(n, 3))).cuda()
    want = rg.barcodes(x, 0).bars
    torch.cuda.synchronize()

    def loop(done):
        for _ in range(ROUNDS):
            assert np.array_equal(rg.barcodes(x, 0).bars, want)
    return loop


def _noalloc_calls(n):
    import torch
    from paper_1908_02518_gb300 import _lib
    lib = _lib.load()
    x = torch.from_numpy(W.distance_matrix(W.cube_points(n, 4))).cuda()
    bars = torch.zeros(n * 32, dtype=torch.uint8, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def loop(done):
        while not done.is_set():
            st = lib.rips_h0_barcode_noalloc(C.c_void_p(x.data_ptr()), n, C.c_float(math.inf), C.c_void_p(bars.data_ptr()),
                                             C.c_void_p(count.data_ptr()), C.c_void_p(stream.cuda_stream))
            assert st == 0, st
            stream.synchronize()
            assert int.from_bytes(count.cpu().numpy().tobytes(), "little") == n
    return loop


def _plan_runs(n):
    import torch
    import paper_1908_02518_gb300 as rg
    x = torch.from_numpy(W.cube_points(n, 5)).cuda()
    plan = rg.BatchPlan([0, n], 3)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    plan.run(x, stream)
    want = plan.result(stream).bars

    def loop(done):
        while not done.is_set():
            plan.run(x, stream)
            assert np.array_equal(plan.result(stream).bars, want)
    return loop


@pytest.mark.parametrize("other", [_noalloc_calls, _plan_runs])
def test_a_smaller_call_beside_a_larger_one(other):
    assert _together(_calls(2000), other(300)) == []
