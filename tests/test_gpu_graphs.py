"""Captured sweep graphs after what they hold by value has changed.

A lattice too large for shared memory replays chunks of sweeps as graphs, whose
phase launches hold the seed's Philox keys: a lattice that gets another seed, by
any of the four calls that give it one, must sweep on that seed's streams.  A batch's
lock-step groups replay graphs too, whose recounts hold the members' histograms: those
enabled between two sweeps of the batch must be the ones that the second one fills.
"""
import os

import numpy as np
import pytest

import oracle

from .gpu_util import first_difference, oracle_run

pytestmark = pytest.mark.gpu

PARAMS = (1 / 0.8, 0.1, 1.0, 0.5)


@pytest.fixture(scope="module")
def cc():
    import paper_2301_11735_gb300 as cc

    return cc


def _phase_lattice(cc, Lx, Ly, **kw):
    """A lattice swept a launch a phase, whatever its size."""
    os.environ["CCMC_NO_RESIDENT"] = "1"
    try:
        return cc.Lattice(Lx, Ly, **kw)
    finally:
        del os.environ["CCMC_NO_RESIDENT"]


@pytest.mark.parametrize("how", ["init_constrained", "init_counts", "set_state",
                                 "set_state_packed"])
@pytest.mark.parametrize("shape", [(64, 32), (68, 36)])
def test_reseeded_lattice_sweeps_on_the_new_seed(cc, shape, how):
    Lx, Ly = shape
    old, new = 11, (7 << 32) | 5
    with _phase_lattice(cc, Lx, Ly) as lat:
        lat.init_constrained(old, 0.1, 0.3)
        lat.sweep(16, *PARAMS)  # captures a chunk of 16
        lat.sweep(16, *PARAMS, obs_every=4)  # and one with records
        done = 0
        if how == "init_constrained":
            lat.init_constrained(new, 0.1, 0.3)
            st = oracle.init_constrained(Lx, Ly, new, 0.1, 0.3)
        elif how == "init_counts":
            lat.init_counts(new, 300, 200)
            st = lat.get_state()
        else:
            st, done = lat.get_state(), 32
            if how == "set_state":
                lat.set_state(st, new, done)
            else:
                lat.set_state_packed(lat.get_state_packed(), new, done)
        for every in (0, 4):
            lat.sweep(16, *PARAMS, obs_every=every)
            st, rec = oracle_run(st, new, done, 16, *PARAMS, obs_every=every)
            done += 16
            got = lat.get_state()
            assert np.array_equal(got, st), (shape, how, every, first_difference(got, st))
        assert np.array_equal(lat.obs_series(), rec)


@pytest.mark.parametrize("enabled", [[0, 1], [5, 12], range(13)])
def test_lock_step_group_fills_the_histograms_enabled_since(cc, enabled):
    shapes = [(256, 64)] * 6 + [(192, 128)] * 7  # enough for a group, rows of whole words
    lats, ref = [], []
    for i, (Lx, Ly) in enumerate(shapes):
        for group in (lats, ref):
            lat = _phase_lattice(cc, Lx, Ly, obs_capacity=64)
            lat.init_constrained(20 + i, 0.1, 0.3)
            group.append(lat)
    with cc.Batch(lats) as b:
        b.config(256, 1024, 2)
        for nbins in (0, 16, 40):  # captured without histograms, then replayed with them
            for i in enabled:
                if nbins:
                    lats[i].hist_enable(nbins)
                    ref[i].hist_enable(nbins)
            for _ in range(2):
                b.sweep(16, *PARAMS, obs_every=2)
            b.sync()
            for i, (lat, one) in enumerate(zip(lats, ref)):
                one.sweep(32, *PARAMS, obs_every=2)
                if nbins and i in enabled:
                    assert lat.hist().sum() == 3 * 16, (nbins, i)
                    assert np.array_equal(lat.hist(), one.hist()), (nbins, i)
    for lat, one in zip(lats, ref):
        assert np.array_equal(lat.get_state(), one.get_state())
        assert np.array_equal(lat.obs_series(), one.obs_series())
        lat.close()
        one.close()
