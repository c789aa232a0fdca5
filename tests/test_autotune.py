"""What the autotuner makes of its probes (given ones here: no GPU): a batch stays on
the library's own plan where no candidate is faster, the fastest candidate is returned
either way, and times taken with other kernels are not used again.  On the GPU: batches
that stay on the plan, go back to it and leave it."""
import numpy as np
import pytest

from paper_2301_11735_gb300 import autotune

SHAPES = [(512, 512)] * 3


@pytest.fixture
def probes(monkeypatch, tmp_path):
    monkeypatch.setattr(autotune, "_CACHE", str(tmp_path / "tune.json"))
    calls = []

    def given(times):
        monkeypatch.setattr(autotune, "_probe", lambda *a: calls.append(a) or dict(times))
        return calls

    return given


@pytest.mark.parametrize("plan,best", [(1.0, 2.0), (2.0, 1.0), (1.0, 1.0)])
def test_the_plan_competes_with_the_candidates(probes, plan, best):
    fast, slow = autotune.CANDIDATES[3], autotune.CANDIDATES[5]
    probes({None: plan, slow: 3.0, fast: best})
    m = autotune.measured(SHAPES)
    assert m["plan"] == (plan <= best)
    assert tuple(m["config"]) == autotune.tune(SHAPES) == fast


def test_times_of_other_kernels_are_taken_again(probes, monkeypatch):
    calls = probes({None: 1.0, autotune.DEFAULT: 2.0})
    for digest, probed in (("a", 1), ("a", 1), ("b", 2), ("a", 2)):
        monkeypatch.setattr(autotune, "_sources", lambda: digest)
        assert autotune.tune(SHAPES) == autotune.DEFAULT
        assert len(calls) == probed
    assert autotune.measured(SHAPES[:2])["plan"] and len(calls) == 3


def test_a_copy_without_the_sources_tunes_as_well(probes, monkeypatch, tmp_path):
    here = autotune._sources()
    monkeypatch.setattr(autotune, "_HERE", str(tmp_path / "elsewhere"))
    probes({None: 1.0, autotune.DEFAULT: 2.0})
    assert autotune.tune(SHAPES) == autotune.DEFAULT and autotune._sources() != here


def test_a_gpu_that_takes_no_candidate_keeps_the_plan(probes):
    calls = probes({None: 1.0})
    assert autotune.measured(SHAPES)["plan"] and autotune.tune(SHAPES) == autotune.DEFAULT
    assert len(calls) == 2  # nothing to keep


@pytest.mark.gpu
def test_tuned_batches_keep_or_return_to_the_plan(probes):
    import paper_2301_11735_gb300 as cc

    given = (256, 4096, 2, 4)
    probes({None: 1.0, given: 2.0})
    params, shapes = (1 / 0.7, 0.2, 1.0, 0.5), [(512, 512)] * 10 + [(64, 64)] * 2
    lats, ref = [], []
    for i, (Lx, Ly) in enumerate(shapes):
        for group in (lats, ref):
            group.append(cc.Lattice(Lx, Ly))
            group[-1].init_constrained(30 + i, 0.1, 0.3)
    with cc.Batch(lats) as b:
        b.sweep(3, *params)
        for config in (None, given):
            if config:
                b.config(*config)
                b.sweep(2, *params)
            assert b.autotune() == given and b.configured is None
            b.sweep(5, *params)
        probes({None: 2.0, given: 1.0})
        autotune._store({})
        assert b.autotune() == given == b.configured
        b.sweep(4, *params)
        b.sync()
    for lat, one in zip(lats, ref):
        one.sweep(19, *params)
        assert np.array_equal(lat.get_state(), one.get_state())
        lat.close()
        one.close()
