"""Batched MD steps on the caller's streams: work on one replica follows a batch
call on the stream that the call used, and the calls can stand in a caller's own
stream capture, with the step and friction that they were given."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2109_07527_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KEYS = ("id", "xyz", "vel")


@pytest.fixture(scope="module")
def crmc():
    from paper_2109_07527_gb300 import crmc as m
    m._lib()
    return m


def _batch(crmc, stream=None):
    s = C.c_void_p(stream.cuda_stream) if stream else None
    return crmc.Batch([crmc.Context(W.config2(seed=7 + r, scale=0.5), stream=s) for r in range(2)])


def _same(a, c):
    for x, y in zip(a.contexts, c.contexts):
        sx, sy = x.state(), y.state()
        for k in KEYS:
            assert np.array_equal(sx[k], sy[k]), k


def test_a_replica_follows_the_stream_of_the_last_batch_call(crmc):
    """The first replica's stream changes between the two halves of a step; the second's velocities are read while
    the closing half waits on the new stream behind 50 ms of other work."""
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    a, ref = _batch(crmc, first), _batch(crmc)
    for b in (a, ref):
        b.md_step(1, 0.005, 1.0, 3)
        b.md_begin(0.005, 1.0, 4)
    torch.cuda.synchronize()
    crmc._lib().cr_set_stream(a.contexts[0]._h, C.c_void_p(second.cuda_stream))
    with torch.cuda.stream(second):
        torch.cuda._sleep(100_000_000)
    a.md_end(0.005, 1.0, 4)
    ref.md_end(0.005, 1.0, 4)
    x, y = a.contexts[1].state(), ref.contexts[1].state()
    for k in KEYS:
        assert np.array_equal(x[k], y[k]), k
    a.close()
    ref.close()


@pytest.mark.parametrize("warm", [False, True])
def test_batched_steps_in_a_callers_capture(crmc, warm):
    """Without friction a step draws no noise that enters the forces, so a replayed step is the step: one captured
    at 0.005 stays that after another at 0.002 was run.  warm: whether steps were taken before the capture."""
    s = torch.cuda.Stream()
    a, ref = _batch(crmc, s), _batch(crmc)
    if warm:
        a.md_step(1, 0.005, 0.0, 3)
        ref.md_step(1, 0.005, 0.0, 3)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.md_step(2, 0.005, 0.0, 9)
    with torch.cuda.stream(s):
        if warm:
            a.md_step(1, 0.002, 0.0, 5)
            ref.md_step(1, 0.002, 0.0, 5)
        g.replay()
    ref.md_step(2, 0.005, 0.0, 9)
    torch.cuda.synchronize()
    _same(a, ref)
    a.close()
    ref.close()
