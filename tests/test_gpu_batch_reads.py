"""Packed reads of small replicas, whose ions are expected to fit one tile of the
ranking, when they do and when one of them has grown past it since."""
import numpy as np
import pytest

from test_gpu_forms import _ions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crmc():
    from paper_2109_07527_gb300 import crmc as m
    m._lib()
    return m


def _read_equals_contexts(b, S):
    R = len(b.contexts)
    n = np.zeros(R, np.int64)
    arr = dict(xyz=np.zeros((R * S, 3), np.float32), vel=np.zeros((R * S, 3), np.float32), id=np.zeros(R * S, np.uint64),
               type=np.zeros(R * S, np.int32))
    b.state_packed(S, arr, n)
    for r, c in enumerate(b.contexts):
        s = c.state()
        assert n[r] == s["n"]
        for key, a in arr.items():
            assert np.array_equal(a[r * S:r * S + n[r]], s[key]), (r, key)
    return n


@pytest.mark.parametrize("ions", [0, 1, 40, 1023, 1024, 1025, 3000])
def test_packed_reads_follow_a_replica_that_grows(crmc, ions):
    w = _ions(200, 40.0, 10.0, 3)
    w.capacity = 4096
    b = crmc.Batch([crmc.Context(w) for _ in range(3)])
    for _ in range(2):
        assert list(_read_equals_contexts(b, w.capacity)) == [200] * 3
    ctx = b.contexts[1]
    ck = ctx.checkpoint()
    if ions:
        rng = np.random.default_rng(ions)
        pairs = ions + ions % 2  # (neutral)
        e = _ions(pairs, 40.0, 10.0, 4)
        new = np.uint64(1 << 32) * np.uint64(2) + rng.permutation(pairs).astype(np.uint64)
        ck.update(n=w.n + pairs, id=np.concatenate([ck["id"], new]), xyz=np.concatenate([ck["xyz"], e.xyz]),
                  vel=np.concatenate([ck["vel"], e.vel]), force=np.zeros((w.n + pairs, 3), np.float32),
                  type=np.concatenate([ck["type"], e.type]), cls=np.concatenate([ck["cls"], e.cls]),
                  state=np.concatenate([ck["state"], e.state]), sweep=8)
    ctx.restore(ck)
    for _ in range(3):
        assert _read_equals_contexts(b, w.capacity)[1] == 200 + ions + ions % 2
    b.close()
