"""The colour phase's chain, however a domain is run.

  * the statistics of unlogged sweeps are those of the trials' records, also
    where consecutive selections scan no list (a box of salt moves);
  * a trial's energy has the same bits wherever the domain's list and halo lie
    (shared or global memory), and logged sweeps give the unlogged chain;
  * the Ewald sums keep the bits they had before the reciprocal vectors went by
    columns, and one box's slices give what a batch's items give;
  * a surrogate runs beside lists that take all of an SM's shared memory;
  * domains of as many cells as ever fitted are accepted;
  * every form of the launch can be named, and gives one chain, with lists and
    halos on chip and in global memory; a form read back can be set again.
"""
import zlib

import numpy as np
import pytest

from paper_2109_07527_gb300 import workloads as W
from parity_util import compare_logs, compare_states
from test_gpu_forms import _electrolyte, _ions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crmc():
    from paper_2109_07527_gb300 import crmc as m
    m._lib()
    return m


def _counts(log):
    acc = (log["flags"] & 1) != 0
    return np.bincount(log["move"], minlength=6)[:6], np.bincount(log["move"][acc], minlength=6)[:6]


@pytest.mark.parametrize("threads", [32, 64, 256, 0])
@pytest.mark.parametrize("n", [2, 800])
def test_statistics_of_salt_moves_are_those_of_the_records(crmc, threads, n):
    """Two ions: most insertions follow one another without a list scan.  threads 0: the tuner's forms, groups of
    one warp among them."""
    a, c = [crmc.Context(_ions(n, 40.0, 10.0, 5, trials_per_domain=24)) for _ in range(2)]
    if threads:
        a.set_launch_shape(threads, 0)
    k = a.trials_per_sweep * 26
    st = a.sweep(k, 9, stats=True)["stats"]
    log = c.sweep(k, 9, log=True)["log"]
    attempts, accepts = _counts(log)
    assert st["trials"] == k
    assert np.array_equal(st["attempts"], attempts) and np.array_equal(st["accepts"], accepts)
    x, y = a.state(), c.state()
    for key in ("id", "xyz", "vel"):
        assert np.array_equal(x[key], y[key]), key
    a.close()
    c.close()


CAPACITIES = [dict(list_capacity=8, halo_capacity=64), dict(list_capacity=4, halo_capacity=32)]


@pytest.mark.parametrize("scale,seed", [(1.0, 11), (0.5, 3)])
def test_energies_do_not_depend_on_where_the_particles_lie(crmc, scale, seed):
    """Every record of the sweeps equal bit for bit (dE and the gross sum S among them): lists and halos on chip
    against both in global memory; flat regions (the full box) and regions compared by minimum images."""
    w = W.config2(seed=seed, scale=scale)
    logs = []
    for kw in [{}] + CAPACITIES:
        g = crmc.Context(w, **kw)
        logs.append(g.sweep(g.trials_per_sweep * 3, 17, log=True)["log"])
        g.close()
    for l in logs[1:]:
        assert logs[0].tobytes() == l.tobytes()


@pytest.mark.parametrize("kw", [{}] + CAPACITIES)
def test_logged_sweeps_give_the_unlogged_chain(crmc, kw):
    w = W.config2(seed=12)
    a, c = [crmc.Context(w, **kw) for _ in range(2)]
    for k in range(3):
        a.sweep(a.trials_per_sweep * 4, 40 + k)
        c.sweep(c.trials_per_sweep * 4, 40 + k, log=True)
    x, y = a.state(), c.state()
    for key in ("id", "xyz", "vel", "state"):
        assert np.array_equal(x[key], y[key]), key
    a.close()
    c.close()


def test_ewald_sums_keep_their_rounding(crmc):
    """Checksums of energies and forces from the version that gave each reciprocal vector a thread (249 particles,
    about 1,500 vectors): sums of float products, so one product fused otherwise shows."""
    w = W.weak_acid_electrolyte(n_acid=150, L=30.0, pH=7.0, pKa=6.5, pIS=1.5, rc=12.0, seed=3, trials_per_domain=40,
                                alpha=0.3)
    w.params["ewald_kmax"] = 9
    g = crmc.Context(w)
    log = np.concatenate([g.sweep(40, 100 + k, log=True)["log"] for k in range(4)])
    assert zlib.crc32(np.ascontiguousarray(log["dE"]).tobytes()) == 0x95a45c54
    g.close()
    g = crmc.Context(w)
    g.sweep(400, 1)
    g.sweep(40, 2, log=True)
    g.md_forces()
    force = g.state()["force"]
    assert force.shape == (249, 3) and zlib.crc32(np.ascontiguousarray(force).tobytes()) == 0x58c73e94
    g.close()


@pytest.mark.parametrize("boxes", [2, 12, 64])
def test_many_ewald_boxes_equal_single_ones(crmc, boxes):
    """64 boxes of 16 reciprocal vectors per axis go by items of a column, well past two CTAs of items per SM; few
    take a vector per thread, and their forces one, two or four particles per CTA."""
    make = lambda r: _electrolyte(20.0, 16, 10 + r, acids=12)
    b = crmc.Batch([crmc.Context(make(r)) for r in range(boxes)])
    b.md_begin(0.005, 1.0, 7)
    b.sweep(2, 50)
    b.md_end(0.005, 1.0, 7)
    for r in (0, boxes // 2, boxes - 1):
        g = crmc.Context(make(r))
        g.md_begin(0.005, 1.0, 7 ^ (r << 32))
        g.sweep(g.trials_per_sweep * 2, 50 ^ (r << 32))
        g.md_end(0.005, 1.0, 7 ^ (r << 32))
        x, y = b.contexts[r].state(), g.state()
        for key in ("id", "xyz", "vel", "state"):
            assert np.array_equal(x[key], y[key]), (r, key)
        g.close()
    b.close()


@pytest.mark.parametrize("threads", [0, 128, 512])
def test_surrogates_run_beside_lists_as_large_as_an_sm(crmc, threads):
    """Every form of a delayed-acceptance sweep fits, logged or not, fixed or tuned, in contexts and in batches (by
    colour and persistent), and gives the chain of small lists."""
    w = W.config2(seed=9, scale=0.5)
    mlp = W.random_mlp(seed=4, gain=0.7, out_gain=0.3)

    def make(**kw):
        g = crmc.Context(w, cell_capacity=512, **kw)
        g.set_surrogate(mlp)
        if threads:
            g.set_launch_shape(threads, 0)
        return g

    large = dict(list_capacity=3091, halo_capacity=64)  # (what 512 threads without a surrogate leave)
    a, ref = make(**large), make()
    n = a.trials_per_sweep * 2
    r = [g.sweep_da(n, 5, log=True)["log"] for g in (a, ref)]
    assert r[0].tobytes() == r[1].tobytes()
    for g in (a, ref):
        g.sweep_da(n * 6, 6)
    for mode in (0, 1):
        b = crmc.Batch([make(**large)])
        b.set_persistent(mode)
        if threads:
            b.set_launch_shape(threads, 0)
        b.sweep_da(2, 5)
        b.sweep_da(12, 6)
        for c in b.contexts + [a]:
            x, y = c.state(), ref.state()
            for key in ("id", "xyz", "vel", "state"):
                assert np.array_equal(x[key], y[key]), key
        b.close()


@pytest.mark.parametrize("cells,per_rc,L,rc", [(19, 2, 57.2, 3.0), (20, 1, 80.5, 2.0)])
def test_domains_of_many_cells(crmc, cells, per_rc, L, rc):
    """The cell tables of 6,859 and 8,000 cells and their halos take nine tenths of an SM's shared memory."""
    w = _ions(400, L, rc, 6, cells_per_rc=per_rc)
    g = crmc.Context(w, domain_cells=cells)
    assert g.info["nc"] == 2 * cells
    n = g.trials_per_sweep * 6
    o, lo, ties = compare_logs(w, g.sweep(n, 8, log=True)["log"], n, 8, dict(domain_cells=cells))
    compare_states(g, o, w.n_sites)
    g.close()


def _code(seats, groups, wide, compact):
    """The second value of a form's pair (cr_set_launch_shape)."""
    return seats | groups << 4 | compact << 8 | wide << 12


# the forms that the tuner chooses among, beyond whole CTAs with the full capacities
FORMS = [(64, _code(1, 1, 16, 1)), (128, _code(1, 4, 16, 0)), (256, _code(1, 8, 16, 0)), (128, _code(2, 1, 2, 0)),
         (256, _code(4, 1, 1, 0)), (256, _code(4, 1, 2, 0)), (256, _code(4, 1, 4, 0)), (256, _code(2, 1, 2, 0)),
         (512, _code(4, 1, 4, 0))]
BOXES = [lambda: W.config2(seed=21, pH=6.0), lambda: W.config4(seed=4, n_rep=1, hi=300)[0],
         lambda: _ions(2400, 40.0, 10.0, 8, clump=0.3)]  # flat; small; lists of 30 to 500 entries


@pytest.fixture(scope="module")
def chains(crmc):
    """The boxes' states after eight sweeps of 128 threads per domain."""
    out = []
    for box in BOXES:
        g = crmc.Context(box())
        g.set_launch_shape(128, 0)
        g.sweep(g.trials_per_sweep * 8, 3)
        out.append(g.state())
        g.close()
    return out


@pytest.mark.parametrize("kw", [{}] + CAPACITIES)
@pytest.mark.parametrize("threads,regs", FORMS + [(32, 0), (512, 0)])
def test_every_form_gives_one_chain(crmc, chains, threads, regs, kw):
    for box, ref in zip(BOXES, chains):
        g = crmc.Context(box(), **kw)
        g.set_launch_shape(threads, regs)
        assert g.launch_shape() == (threads, regs)
        g.sweep(g.trials_per_sweep * 8, 3)
        s = g.state()
        for key in ("id", "xyz", "vel", "state"):
            assert np.array_equal(s[key], ref[key]), key
        g.close()


def test_a_tuned_form_can_be_read_and_set_again(crmc):
    g, c = [crmc.Context(W.config2(seed=21, scale=0.5)) for _ in range(2)]
    b = crmc.Batch([c])
    for x, k in ((g, g.trials_per_sweep * 30), (b, 60)):
        x.sweep(k, 1)
        shape = x.launch_shape()
        assert shape in FORMS + [(t, 0) for t in (128, 256, 512)]
        x.set_launch_shape(128, 4)
        assert x.launch_shape() == (128, 4)
        x.set_launch_shape(*shape)
        assert x.launch_shape() == shape
    for bad in ((256, 17), (64, _code(4, 1, 2, 0)), (128, -1), (96, 0)):
        with pytest.raises(crmc.CrError):
            g.set_launch_shape(*bad)
        with pytest.raises(crmc.CrError):
            b.set_launch_shape(*bad)
    b.close()
