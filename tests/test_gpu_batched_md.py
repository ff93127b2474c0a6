"""Batched MD steps, the forces' fixed-point terms, the Ewald kernels' layouts.

  * cr_md_forces (each pair once, the flat frame, the partner's share by
    atomics) gives the bits of cr_md_forces_noalloc (every pair from both
    ends): few and many cells per dimension, one and two cells per cutoff,
    dense corners, terms beyond an int's range, a WCA cutoff beyond the Coulomb
    cutoff;
  * a batched MD step (one launch for all replicas) gives the bits of the
    contexts' own steps, for replicas of unequal size, with and without Ewald
    electrostatics, and after one replica has been stepped by itself;
  * S(k) and its forces do not depend on how the vectors are dealt to threads;
  * a force evaluation of more particles than the capacity is refused.
"""
import numpy as np
import pytest

from paper_2109_07527_gb300 import workloads as W
from test_zz_no_alloc import _check, _noalloc, _slots

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


LONG = dict(wca_del=[0.0] * 5 + [6.0] + [0.0] * 10)  # class 1 pairs: cutoff 6 + 2^(1/6)


@pytest.mark.parametrize("n,L,rc,clump,kw", [
    (2, 40.0, 10.0, 0.0, {}),                                    # nearly every cell empty
    (600, 20.0, 10.0, 0.0, {}),                                  # 4 cells per dimension: each once
    (800, 27.5, 10.0, 0.0, dict(schedule=1)),                    # 5 cells: the stencil is the box
    (800, 33.0, 10.0, 0.0, dict(schedule=1)),                    # 6
    (800, 37.0, 10.0, 0.0, dict(schedule=1)),                    # 7
    (1500, 60.0, 10.0, 0.0, {}),                                 # 12 cells
    (3000, 60.0, 10.0, 0.3, {}),                                 # a dense corner across the boundary
    (6000, 40.0, 10.0, 0.5, dict(cells_per_rc=1, domain_cells=1)),
    (1200, 60.0, 6.0, 0.2, LONG),                                # 20 cells, partners beyond the stencil left out
    (500, 24.0, 6.0, 0.0, LONG),
])
def test_forces_once_per_pair_equal_those_from_both_ends(crmc, n, L, rc, clump, kw):
    torch = pytest.importorskip("torch")
    ctx = crmc.Context(_ions(n, L, rc, 7 + n, clump, **kw))
    for _ in range(2):  # the sums of the first evaluation are gone
        ctx.md_forces()
    ref = ctx.state()
    assert np.abs(ref["force"]).max() > 0 or n < 10
    force, ids = _noalloc(torch, ctx, _slots(ctx))
    _check(ref, force, ids)
    ctx.close()


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


@pytest.mark.parametrize("alone", [False, True])
@pytest.mark.parametrize("kind", ["ragged", "ewald"])
def test_batched_md_equals_single_contexts(crmc, kind, alone):
    make = (lambda: W.config4(seed=5, n_rep=4, hi=400)) if kind == "ragged" else (
        lambda: [_electrolyte(20.0, 6, 1), _electrolyte(26.0, 0, 2), _electrolyte(30.0, 9, 3)])
    a = [crmc.Context(w) for w in make()]
    c = [crmc.Context(w) for w in make()]
    b = crmc.Batch(a)
    if alone:  # the replicas' evaluation counters differ from here on
        a[1].md_step(1, 0.005, 1.0, 77)
        c[1].md_step(1, 0.005, 1.0, 77)
    b.md_step(2, 0.005, 1.0, 11)
    for k, dt in ((0, 0.005), (1, 0.005), (2, 0.004)):
        b.md_begin(dt, 1.0, 40 + k)
        b.sweep(1, 50 + k)
        b.md_end(dt, 1.0, 40 + k)
    for r, g in enumerate(c):
        g.md_step(2, 0.005, 1.0, 11 ^ (r << 32))
        for k, dt in ((0, 0.005), (1, 0.005), (2, 0.004)):
            g.md_begin(dt, 1.0, (40 + k) ^ (r << 32))
            g.sweep(g.trials_per_sweep, (50 + k) ^ (r << 32))
            g.md_end(dt, 1.0, (40 + k) ^ (r << 32))
    _same(a, c)
    b.close()


def test_ewald_items_and_slices_give_the_same_chain(crmc):
    """31 replicas of |n| <= 16 fill the GPU with items of four |nz|, a single context takes one |nz| per thread."""
    ws = [_electrolyte(20.0 + 0.1 * r, 16, r, acids=10) for r in range(31)]
    a = [crmc.Context(w) for w in ws]
    b = crmc.Batch(a)
    b.sweep(2, 9)
    b.md_step(1, 0.005, 1.0, 3)
    c = []
    for r in (0, 17, 30):
        g = crmc.Context(ws[r])
        g.sweep(g.trials_per_sweep * 2, 9 ^ (r << 32))
        g.md_step(1, 0.005, 1.0, 3 ^ (r << 32))
        c.append(g)
    _same([a[0], a[17], a[30]], c)
    b.close()


def test_forces_beyond_the_capacity_are_refused(crmc):
    """An electrolyte of acids alone sets its counter-ions free: more particles than its capacity after a sweep."""
    w = W.weak_acid_electrolyte(n_acid=300, L=60.0, pH=9.0, pKa=5.0, pIS=2.0, rc=15.0, seed=2, trials_per_domain=400)
    w.capacity = w.n
    ctx = crmc.Context(w)
    ctx.sweep(ctx.trials_per_sweep, 3)
    assert ctx.counts()["n"] > w.n
    with pytest.raises(crmc.CrError) as e:
        ctx.md_forces()
    assert e.value.code == -4  # CR_ERR_CAPACITY
    ctx.close()
