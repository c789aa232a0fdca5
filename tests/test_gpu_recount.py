"""The recount kernel's launch shapes against the oracle's recount: quads of words in
blocks of 256 (less than a wave) and of 1024 threads (8192 x 5120 is the first whole
quad size of 8192 columns above the line), with a record and histograms."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly", [(256, 16), (8192, 4096), (8192, 5120)])
def test_recount_matches_oracle(Lx, Ly):
    import paper_2301_11735_gb300 as cc

    with cc.Lattice(Lx, Ly, obs_capacity=2) as lat:
        lat.init_constrained(11, 0.1, 0.3)
        lat.hist_enable(16)
        lat.sweep(1, 0.8, 0.2, 1.0, 0.5, obs_every=1)
        record = lat.obs_series(cap=2)[0]
        now = lat.observables()
        hist = lat.hist()
        expected = list(oracle.recount(lat.get_state()))
    keys = ("Nc", "BV", "BJ", "M", "M_stag", "S_sum", "S_stag")
    assert [int(now[k]) for k in keys] == [int(x) for x in expected]
    assert [int(x) for x in record[1:8]] == [int(x) for x in expected]
    N = Lx * Ly
    for h, k in enumerate((3, 4, 6)):  # M, M_stag, S_stag
        want = np.zeros(16, dtype=np.int64)
        want[(int(expected[k]) + N) * 16 // (2 * N + 1)] = 1
        assert (hist[h] == want).all()
