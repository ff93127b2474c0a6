"""Batched MD steps on the caller's streams: the calls can stand in a caller's own
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
