"""How lattices are held in shared memory where the GPU places clusters of 16, 8,
4, 2 or no CTAs (a part of a GPU may not have sixteen SMs side by side): the plan
itself, on the CPU, and the sweeps of a device without clusters.
"""
import itertools

import numpy as np
import pytest

import oracle
import paper_2301_11735_gb300 as cc

from .gpu_util import first_difference, oracle_run

LIMITS = (0, 1, 2, 4, 8, 16)
SIDES = (4, 8, 12, 16, 36, 60, 64, 68, 128, 132, 252, 256, 260, 516, 768, 1000, 1024, 1072, 2052,
         4096, 16384, 131072)
MAX_SMEM = 224 << 10


@pytest.mark.parametrize("limit", LIMITS)
def test_plans_fit_the_device(limit):
    for Lx, Ly in itertools.product(SIDES, SIDES):
        if Lx * Ly > 1 << 30:
            continue
        p = cc.resident_plan(Lx, Ly, limit)
        W, Cy = (Lx // 4 + 15) // 16, Ly // 4
        if p["ctas"] == 0:
            continue
        assert p["ctas"] <= limit and p["ctas"] in LIMITS, (Lx, Ly, p)
        assert p["rows"] * p["ctas"] >= Cy and 64 * p["rows"] * W < p["smem"] <= MAX_SMEM
        assert p["ctas"] == 1 or p["rows"] >= 2  # row numbers are divided by multiplication
        assert p["threads_per_word"] in (1, 2, 4)
    assert (cc.resident_plan(16, 16, limit)["ctas"] == 0) == (limit == 0)


def test_plans_refuse_what_is_no_lattice_or_limit():
    for args in ((6, 8, 16), (8, 2, 16), (64, 64, 3), (64, 64, 32), (64, 64, -1)):
        with pytest.raises(cc.CcmcError) as e:
            cc.resident_plan(*args)
        assert e.value.code == cc.E_INVAL


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(256, 256), (260, 516), (768, 512), (1000, 1000)])
def test_lattices_of_a_device_without_clusters(shape, monkeypatch):
    """One CTA, or a launch a phase where one does not hold the lattice; alone and
    in batches, whose limit of sites may hold more than ccmc_sweep would."""
    Lx, Ly = shape
    assert cc.resident_plan(Lx, Ly)["ctas"] > 1 >= cc.resident_plan(Lx, Ly, 1)["ctas"]
    monkeypatch.setenv("CCMC_FAULT", "cluster")
    lats = [cc.Lattice(Lx, Ly, obs_capacity=16) for _ in range(3)]
    monkeypatch.delenv("CCMC_FAULT")
    params = (1 / 0.7, 0.2, 1.0, 0.5)
    st = oracle.init_constrained(Lx, Ly, 8, 0.1, 0.3)
    for lat in lats:
        lat.init_constrained(8, 0.1, 0.3)
    lats[0].sweep(7, *params, obs_every=2)
    for lat, cfg in zip(lats[1:], (None, (256, 200000, 1, 4))):
        with cc.Batch([lat]) as b:
            if cfg:
                b.config(*cfg)
            b.sweep(7, *params, obs_every=2)
            b.sync()
    st, rec = oracle_run(st, 8, 0, 7, *params, obs_every=2)
    for lat in lats:
        got = lat.get_state()
        assert np.array_equal(got, st), (shape, first_difference(got, st))
        assert np.array_equal(lat.obs_series(), rec)
        lat.close()
