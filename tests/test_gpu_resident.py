"""The resident kernel (whole sweeps of a lattice in one launch) at the edges of
its shapes: rows shorter than a word, one row of classes, tails, one CTA with one
or several passes, clusters whose last CTAs own fewer rows or none, the largest
default size; and the per-phase kernels on lattices the resident kernel would
take.  Bit-exact against the oracle, or for the larger ones against the per-phase
path, states, records and histograms alike.
"""
import os

import numpy as np
import pytest

import oracle

from .gpu_util import first_difference, oracle_run

pytestmark = pytest.mark.gpu

PARAMS = (1 / 0.7, 0.2, 1.0, 0.5)


@pytest.fixture(scope="module")
def cc():
    import paper_2301_11735_gb300 as cc

    return cc


def _lattice(cc, Lx, Ly, **env):
    """A lattice created under environment variables that select a path."""
    os.environ.update(env)
    try:
        return cc.Lattice(Lx, Ly, obs_capacity=16)
    finally:
        for k in env:
            os.environ.pop(k)


# one CTA (a word a thread, rows of one site), clusters of 2 to 16 (rows that do
# not divide by the CTAs, words that do not divide by the warps)
SMALL = [(4, 4), (4, 64), (64, 4), (12, 8), (60, 36), (64, 64), (68, 124), (128, 128), (132, 140),
         (192, 256), (256, 260), (2052, 16), (16, 2052)]
LARGE = [(448, 384), (448, 448), (516, 516), (768, 400), (1000, 1000), (1024, 1024), (64, 4096), (4096, 64), (1088, 1084)]
# few rows of classes, so that no shape or only one CTA holds them
WIDE = [(131072, 4), (262144, 4), (131072, 8), (32768, 32)]


@pytest.mark.parametrize("shape", SMALL)
def test_resident_sweeps_match_oracle(cc, shape):
    Lx, Ly = shape
    seed = 40 + Lx + Ly
    st = oracle.init_constrained(Lx, Ly, seed, 0.1, 0.3)
    with _lattice(cc, Lx, Ly) as lat:
        lat.init_constrained(seed, 0.1, 0.3)
        done = 0
        for n, every in ((1, 1), (5, 2), (20, 3)):
            lat.sweep(n, *PARAMS, obs_every=every)
            st, rec = oracle_run(st, seed, done, n, *PARAMS, obs_every=every)
            done += n
            got = lat.get_state()
            assert np.array_equal(got, st), (shape, done, first_difference(got, st))
            assert np.array_equal(lat.obs_series()[-len(rec):], rec), (shape, done)


@pytest.mark.parametrize("shape", LARGE + WIDE)
def test_resident_sweeps_match_the_phase_kernels(cc, shape):
    out = []
    for env in ({}, {"CCMC_NO_RESIDENT": "1"}):
        with _lattice(cc, *shape, **env) as lat:
            lat.hist_enable(32)
            lat.init_constrained(9, -0.05, 0.3)
            lat.sweep(21, *PARAMS, obs_every=2)
            out.append((lat.get_state(), lat.obs_series(), lat.hist()))
    for a, b in zip(*out):
        assert np.array_equal(a, b), (shape, first_difference(a, b))


@pytest.mark.parametrize("shape", [(256, 256), (512, 128), (1024, 64), (36, 44), (260, 36)])
def test_phase_kernels_still_match_oracle_on_small_lattices(cc, shape):
    Lx, Ly = shape
    st = oracle.init_constrained(Lx, Ly, 5, 0.05, 0.3)
    with _lattice(cc, Lx, Ly, CCMC_NO_RESIDENT="1") as lat:
        lat.init_constrained(5, 0.05, 0.3)
        lat.sweep(19, *PARAMS, obs_every=1)  # a replayed graph, then single sweeps
        st, rec = oracle_run(st, 5, 0, 19, *PARAMS)
        assert np.array_equal(lat.get_state(), st)
        assert np.array_equal(lat.obs_series(), rec[-16:])


@pytest.mark.parametrize("cfg", [(64, 200000, 1, 4), (256, 200000, 2, 1), (512, 200000, 8, 4)])
def test_batches_of_every_shape_match_single_sweeps(cc, cfg):
    """Lattices of different shapes (several launches side by side, clusters among
    them), uneven sweeps, twice in a row."""
    shapes = SMALL[:10] + [(256, 260), (516, 260), (400, 400)]
    nsw = [3 + 2 * i for i in range(len(shapes))]
    lats, ref = [], []
    for i, (Lx, Ly) in enumerate(shapes):
        for group in (lats, ref):
            lat = cc.Lattice(Lx, Ly, obs_capacity=16)
            lat.init_constrained(60 + i, 0.1, 0.3)
            group.append(lat)
    with cc.Batch(lats) as b:
        b.config(*cfg)
        for _ in range(2):
            b.sweep(nsw, *PARAMS, obs_every=3)
        b.sync()
    for i, (lat, one) in enumerate(zip(lats, ref)):
        one.sweep(2 * nsw[i], *PARAMS, obs_every=3)
        assert np.array_equal(lat.get_state(), one.get_state()), (cfg, shapes[i])
        assert np.array_equal(lat.obs_series(), one.obs_series()), (cfg, shapes[i])
        lat.close()
        one.close()


@pytest.mark.parametrize("shapes", [[(516, 260)] * 7 + [(260, 1024)] * 6, [(512, 256)] * 13])
def test_lock_step_groups_match_single_sweeps(cc, shapes):
    """Enough lattices beyond the resident limit to advance with one launch a phase."""
    lats, ref = [], []
    for i, (Lx, Ly) in enumerate(shapes):
        for group in (lats, ref):
            lat = cc.Lattice(Lx, Ly, obs_capacity=16)
            lat.init_constrained(80 + i, 0.1, 0.3)
            group.append(lat)
    T = [0.3 + 0.2 * i for i in range(len(shapes))]
    with cc.Batch(lats) as b:
        b.config(256, 1024, 2)
        for _ in range(2):  # the second call replays the captured group graph
            b.sweep(18, [1 / t for t in T], 0.1, 0.5, 1.0, obs_every=2)
        b.sync()
    for lat, one, t in zip(lats, ref, T):
        one.sweep(36, 1 / t, 0.1, 0.5, 1.0, obs_every=2)
        assert np.array_equal(lat.get_state(), one.get_state())
        assert np.array_equal(lat.obs_series(), one.obs_series())
        lat.close()
        one.close()
