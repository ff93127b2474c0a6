"""The colour phase's chain, however a domain is run.

  * the statistics of unlogged sweeps are those of the trials' records, also
    where consecutive selections scan no list (a box of salt moves);
  * a trial's energy has the same bits wherever the domain's list and halo lie
    (shared or global memory), and logged sweeps give the unlogged chain.
"""
import numpy as np
import pytest

from paper_2109_07527_gb300 import workloads as W
from test_gpu_forms import _ions

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
