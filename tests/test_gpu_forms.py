"""The colour phase's forms, shapes of mixed batches, reads of many inserted ions.

  * every form that the tuner may pick (threads, seats, groups, compact
    capacities; persistent or by colour) gives the same chain;
  * a batch whose largest list and largest region belong to different replicas
    is accepted and runs each replica's own chain;
  * a surrogate layer gives the same values at every thread count;
  * a read ranks inserted ions within tiles of 1024 and across them.
"""
import numpy as np
import pytest

from paper_2109_07527_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crmc():
    from paper_2109_07527_gb300 import crmc as m
    m._lib()
    return m


def _ions(n, L, rc, seed, clump=0.0, **kw):
    """n ions (and, with a class 1 pair table, cores among them) at random, a part of them in one corner."""
    rng = np.random.default_rng(seed)
    x = rng.random((n, 3)) * L
    k = int(clump * n)
    x[:k] = np.mod(rng.normal(size=(k, 3)) * 2.0, L)
    x = x.astype(np.float32)
    x[x >= np.float32(L)] = 0.0
    kinds = np.where(np.arange(n) % 2 == 0, W.XP, W.XM).astype(np.int32)
    cls = np.zeros(n, np.int32)
    if "wca_del" in kw:
        kinds[::8], cls[::8] = W.CORE, 1
        kinds[1::8], cls[1::8] = W.CORE, 1
    return W.Workload(name="ions", xyz=x, type=kinds, cls=cls, state=np.zeros(n, np.int8), pK=np.zeros(n),
                      bonds=np.zeros((0, 2), np.int32), vel=rng.normal(size=(n, 3)).astype(np.float32),
                      params=W.default_params(box_L=L, rc=rc, **kw), capacity=n + 512, meta={})


def _electrolyte(L, kmax, seed, acids=40, rc=8.0):
    w = W.weak_acid_electrolyte(n_acid=acids, L=L, pH=7.0, pKa=6.5, pIS=2.0, rc=rc, seed=seed, trials_per_domain=40,
                                alpha=0.4)
    w.params["ewald_kmax"] = kmax
    return w


def _same(a, c):
    for x, y in zip(a, c):
        sx, sy = x.state(), y.state()
        for k in ("id", "xyz", "vel", "state"):
            assert np.array_equal(sx[k], sy[k]), k


def test_a_batch_of_unequal_boxes_is_accepted(crmc):
    """Lists take what an SM has under the global schedule: a long list beside another replica's larger region
    and reciprocal sum exceeds it, and is cut."""
    ws = [_electrolyte(20.0, 6, 1), _electrolyte(26.0, 0, 2), _electrolyte(30.0, 9, 3)]
    a, c = [[crmc.Context(w) for w in ws] for _ in range(2)]
    b = crmc.Batch(a)
    b.sweep(3, 50)
    for r, g in enumerate(c):
        g.sweep(g.trials_per_sweep * 3, 50 ^ (r << 32))
    _same(a, c)
    b.close()


@pytest.mark.parametrize("ions", [0, 2, 1022, 1024, 1026, 2050])
def test_reads_order_inserted_ions_at_the_tiles_edges(crmc, ions):
    """Ions of ids beyond 2^32 in no particular order: ranked within tiles of 1024 and across them."""
    w = _ions(1500, 40.0, 10.0, 3)
    w.capacity = 4096
    ctx = crmc.Context(w)
    ck = ctx.checkpoint()
    rng = np.random.default_rng(ions)
    e = _ions(ions, 40.0, 10.0, 4) if ions else None
    # (ids as two domain sweeps give them: phase + 1 in the high word)
    new = (np.uint64(1 << 32) * (1 + rng.integers(0, 3, ions)).astype(np.uint64) +
           rng.permutation(max(ions, 1))[:ions].astype(np.uint64))
    if ions:
        ck.update(n=w.n + ions, id=np.concatenate([ck["id"], new]),
                  xyz=np.concatenate([ck["xyz"], e.xyz]), vel=np.concatenate([ck["vel"], e.vel]),
                  force=np.zeros((w.n + ions, 3), np.float32), type=np.concatenate([ck["type"], e.type]),
                  cls=np.concatenate([ck["cls"], e.cls]), state=np.concatenate([ck["state"], e.state]), sweep=8)
    ctx.restore(ck)
    s = ctx.state()
    order = np.argsort(ck["id"], kind="stable")
    assert np.array_equal(s["id"], ck["id"][order])
    assert np.array_equal(s["xyz"], ck["xyz"][order]) and np.array_equal(s["type"], ck["type"][order])
    ctx.close()


def test_every_form_of_the_colour_phase_gives_the_same_chain(crmc):
    """The tuner's rounds run each form in turn (threads, seats, groups, compact capacities; persistent or by
    colour) on the same chain; dense and sparse domains, one small box."""
    make = lambda: [W.config2(seed=21, scale=0.5, pH=p) for p in (3.0, 6.0)] + W.config4(seed=4, n_rep=2, hi=300)
    a, c = [[crmc.Context(w) for w in make()] for _ in range(2)]
    b, f = crmc.Batch(a), crmc.Batch(c)
    f.set_persistent(0)
    f.set_launch_shape(128, 0)
    b.sweep(60, 31)
    f.sweep(60, 31)
    _same(a, c)
    b.close()
    f.close()


@pytest.mark.parametrize("threads", [128, 256])
def test_surrogate_layers_match_at_every_thread_count(crmc, threads):
    """A thread takes an output of both vectors below 256 threads, of one from 256."""
    mlp = W.random_mlp(seed=4, gain=0.7, out_gain=0.3)
    got = []
    for t in (threads, 512):
        g = crmc.Context(W.config2(seed=9, scale=0.5))
        g.set_surrogate(mlp)
        g.set_launch_shape(t, 0)
        g.sweep_da(g.trials_per_sweep * 3, 5)
        got.append(g)
    _same(got[:1], got[1:])
