"""The kernels that run a launch a phase, at the sizes where their launches change:
several rounds of words a CTA (CCMC_TILE_GRID caps the CTAs of a phase), CTAs of 64,
128 and 256 threads, rows of whole words and ragged ones, nearest-neighbour phases,
lock-step groups.  Bit-exact against the oracle, launched directly and replayed.
"""
import os
import time

import numpy as np
import pytest

import oracle

from .gpu_util import first_difference, oracle_run
from .test_gpu_parity import _near_seed

pytestmark = pytest.mark.gpu

PARAMS = (1 / 0.8, 0.1, 1.0, 0.5)


@pytest.fixture(scope="module")
def cc():
    import paper_2301_11735_gb300 as cc

    return cc


def _phase_lattice(cc, Lx, Ly, ctas=0):
    env = {"CCMC_TILE_GRID": str(ctas)} if ctas else {"CCMC_NO_RESIDENT": "1"}
    os.environ.update(env)
    try:
        return cc.Lattice(Lx, Ly, obs_capacity=32)
    finally:
        for k in env:
            del os.environ[k]


def _check(cc, Lx, Ly, ctas=0, seed=77):
    with _phase_lattice(cc, Lx, Ly, ctas) as lat:
        lat.init_constrained(seed, 0.1, 0.3)
        st, done = lat.get_state(), 0
        for n in (2, 16):  # launched directly; replayed
            lat.sweep(n, *PARAMS, obs_every=2)
            st, rec = oracle_run(st, seed, done, n, *PARAMS, obs_every=2)
            done += n
            got = lat.get_state()
            assert np.array_equal(got, st), (Lx, Ly, ctas, n, first_difference(got, st))
        assert np.array_equal(lat.obs_series()[1:], rec)


@pytest.mark.parametrize("ctas", [1, 3])
@pytest.mark.parametrize("shape", [(256, 256), (260, 260), (1004, 64), (1024, 256), (36, 1028)])
def test_several_rounds_of_words_a_cta(cc, shape, ctas):
    _check(cc, *shape, ctas)


def test_the_cap_takes_effect(cc):
    """2048 x 2048: 16384 words of a phase on one CTA take 128 rounds."""
    seconds = []
    for ctas in (0, 1):
        with _phase_lattice(cc, 2048, 2048, ctas) as lat:
            lat.init_constrained(1, 0.1, 0.3)
            lat.phases(8, *PARAMS)
            lat.sync()
            t0 = time.perf_counter()
            lat.phases(40, *PARAMS)
            lat.sync()
            seconds.append(time.perf_counter() - t0)
    assert seconds[1] > 3 * seconds[0], seconds


# 2 words a row: 9728 and 9730 words (CTAs of 64 and 128 threads), 19456 and 19458
# (128 and 256); whole words a row: 9732 and 19460
@pytest.mark.parametrize("shape", [(68, 19456), (68, 19460), (68, 38912), (68, 38916),
                                   (256, 9732), (256, 19460)])
def test_cta_sizes(cc, shape):
    _check(cc, *shape)


@pytest.mark.parametrize("Lx", [1024, 1004])
@pytest.mark.parametrize("dx,dy", [(1, 0), (-1, 0), (0, 1), (0, -1)])
def test_nearest_neighbour_phases(cc, Lx, dx, dy):
    Ly = 64
    seed, P = _near_seed(Lx, Ly, (dx % Lx, dy % Ly))
    nsw = P // 8 + 1
    st = oracle.init_constrained(Lx, Ly, seed, 0.1, 0.4)
    with _phase_lattice(cc, Lx, Ly) as lat:
        lat.init_constrained(seed, 0.1, 0.4)
        lat.sweep(nsw, *PARAMS)
        st, _ = oracle_run(st, seed, 0, nsw, *PARAMS, obs_every=0)
        got = lat.get_state()
        assert np.array_equal(got, st), (dx, dy, seed, P, first_difference(got, st))


@pytest.mark.parametrize("ctas", [0, 3])
@pytest.mark.parametrize("shapes", [[(256, 256)] * 9 + [(512, 64)] * 4,
                                    [(260, 260)] * 6 + [(68, 516)] * 6])
def test_lock_step_groups(cc, shapes, ctas):
    lats = []
    for i, (Lx, Ly) in enumerate(shapes):
        lats.append(_phase_lattice(cc, Lx, Ly, ctas))
        lats[-1].init_constrained(60 + i, 0.1, 0.3)
    with cc.Batch(lats) as b:
        for n in (2, 16):
            b.sweep(n, *PARAMS, obs_every=2)
        b.sync()
    for i, ((Lx, Ly), lat) in enumerate(zip(shapes, lats)):
        st = oracle.init_constrained(Lx, Ly, 60 + i, 0.1, 0.3)
        st, rec = oracle_run(st, 60 + i, 0, 18, *PARAMS, obs_every=2)
        got = lat.get_state()
        assert np.array_equal(got, st), (Lx, Ly, ctas, first_difference(got, st))
        assert np.array_equal(lat.obs_series(), rec)
        lat.close()


def test_largest_lattice_of_one_site_a_word(cc):
    """4 x 2^28 sites take 2^32 bytes: the phase kernel's byte offsets reach 2^32 - 4."""
    Lx, Ly, seed = 4, 1 << 28, 9
    packed = np.random.default_rng(1).integers(0, 256, size=Lx * Ly // 4, dtype=np.uint8)
    st = np.empty((Ly, Lx), np.uint8)
    for k in range(4):
        st[:, k] = (packed >> (2 * k)) & 3
    with cc.Lattice(Lx, Ly) as lat:
        lat.set_state_packed(packed, seed, 0)
        lat.phases(1, *PARAMS)
        got = lat.get_state_packed()
    oracle.phase(st, seed, 0, oracle.threshold_table(*PARAMS))
    assert np.array_equal(got, st[:, 0] | (st[:, 1] << 2) | (st[:, 2] << 4) | (st[:, 3] << 6))
    assert not np.array_equal(got, packed)
