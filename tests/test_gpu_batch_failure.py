"""A batched sweep that fails between its launches (injected on the host) returns when
what it queued has ended: the caller may then destroy the lattices, whose memory goes
to others.  Meanwhile the server goes on serving.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

PARAMS = (1 / 0.7, 0.2, 1.0, 0.5)


def test_failed_batch_call_leaves_nothing_running(monkeypatch):
    import torch

    import paper_2301_11735_gb300 as cc

    stream = torch.cuda.Stream()
    lats = []
    for i, L in enumerate((256, 64, 128)):  # three shapes: three launches
        lat = cc.Lattice(L, L)
        lat.init_constrained(i, 0.1, 0.3)
        lats.append(lat)
    with cc.Batch(lats, stream=stream) as b:
        monkeypatch.setenv("CCMC_FAULT", "group")
        with pytest.raises(cc.CcmcError) as e:
            b.sweep(8000, *PARAMS)  # about 60 ms of the 256 x 256 lattice, queued first
        assert e.value.code == cc.E_CUDA
        assert stream.query()
        monkeypatch.delenv("CCMC_FAULT")
        for lat in lats:
            lat.close()
    for i, L in enumerate((256, 64, 128)):  # the memory is whole again
        with cc.Lattice(L, L) as lat:
            lat.init_constrained(50 + i, 0.1, 0.3)
            st = oracle.init_constrained(L, L, 50 + i, 0.1, 0.3)
            assert np.array_equal(lat.get_state(), st)


def test_server_survives_a_failed_slice(monkeypatch):
    import paper_2301_11735_gb300 as cc

    monkeypatch.setenv("CCMC_FAULT", "group")
    with cc.Server(hbm_budget_bytes=1 << 30) as srv:
        long = [srv.submit(L, L, L, 0.1, 100000, *PARAMS) for L in (64, 256, 128)]
        codes = [srv.wait(t, timeout_s=60.0)["status"] for t in long]
        assert cc.E_CUDA in codes and set(codes) <= {cc.OK, cc.E_CUDA}, codes
        monkeypatch.delenv("CCMC_FAULT")
        out = np.empty(64 * 64, dtype=np.uint8)
        t = srv.submit(64, 64, 7, 0.1, 12, *PARAMS, state_out=out)
        assert srv.wait(t, timeout_s=60.0)["status"] == cc.OK
    st = oracle.init_constrained(64, 64, 7, 0.1, 0.3)
    oracle.sweeps(st, 7, 0, 12, *PARAMS, obs_every=0)
    assert np.array_equal(out.reshape(64, 64), st)
